// bandwidth.cu -- kernel bandwidth selection (Sec. 2.2).
//
// Median rule (Eq. model_bandwidth): h = med / sqrt(2 ln N), med the lower
// middle order statistic of the N(N-1)/2 distances |q_J - q_K|, J < K.  The
// selection is exact on FP32 squared distances (their bit patterns, the keys,
// order like the values), entirely on the device:
//   1. a bracket [lo, hi] of keys around the median from the keys of n random
//      pairs, n = M / 1024 of the M pairs (at least 2^20): the sample's order
//      statistics n/2 -+ 2.5 sqrt(n), five standard deviations away;
//   2. one pass over all unordered pairs (k_bracket) that counts the keys
//      below lo and collects those inside, about 160 sqrt(M) of them;
//   3. an exact radix select among the collected keys.
// Where the bracket misses the median (by the counts of step 2; once in 10^6
// clouds), or the sample shows many equal distances, or a particle lies so far
// out that the screen of step 2 has no resolution, or the keys take more room
// than there is (from about three million particles on), a radix select by three
// histogram passes over all pairs (k_hist) takes over.  Clouds of up to SMALL_PAIRS
// pairs write all keys and select among them.
//
// The FP32 and integer issue bounds step 2.  It screens the pairs by
// |y_i|^2 + |y_j|^2 - 2 y_i.y_j of centred coordinates y (D + 1 operations
// instead of 2D) against the bracket widened by a bound on everything that
// this form can be off by, and forms the key itself only for the few pairs
// inside (those queued for the end of the item, so that no lane waits).  Each
// of the three histogram passes over ordered pairs takes 2 (2D) and a
// shared-memory atomic for most pairs.  N = 65536, D = 9: histograms 14.2 ms,
// bracket without the screen 2.51 ms, with it 1.53 ms
// (k_bracket 1.36).
//
// Silverman rule: h = sigma (4 / ((D+2) N))^(1/(D+4)), sigma the mean over
// coordinates of the sample standard deviation (two FP64 passes).
#include <math.h>

#include <type_traits>

#include "pair.cuh"

namespace {

struct SelState {
  unsigned long long rank;  // rank still to find inside the current prefix
  unsigned prefix;          // key bits selected so far
  unsigned pad;
};

constexpr int BW_NT = 256;
constexpr int NBINS = 2048;

__host__ __device__ constexpr int pass_shift(int pass) { return pass == 0 ? 21 : (pass == 1 ? 10 : 0); }
__host__ __device__ constexpr int pass_bits(int pass) { return pass == 2 ? 10 : 11; }

template <int D>
__global__ void __launch_bounds__(BW_NT)
    k_hist(const float *__restrict__ q, int N, int jchunk, const SelState *__restrict__ st, int pass,
           unsigned long long *__restrict__ ghist) {
  __shared__ unsigned hist[NBINS];
  __shared__ float tile[BW_NT * D];
  const int tid = threadIdx.x;
  const int shift = pass_shift(pass), bits = pass_bits(pass);
  const unsigned mask = (1u << bits) - 1u;
  const int hi = shift + bits;
  const unsigned prefix = st->prefix;
  for (int b = tid; b < NBINS; b += BW_NT) hist[b] = 0u;
  const int i = blockIdx.x * BW_NT + tid;
  const bool vi = i < N;
  float xi[D];
#pragma unroll
  for (int d = 0; d < D; ++d) xi[d] = vi ? q[(size_t)i * D + d] : 0.f;
  const int j0 = blockIdx.y * jchunk;
  const int j1 = min(N, j0 + jchunk);
  for (int jt = j0; jt < j1; jt += BW_NT) {
    const int cnt = min(BW_NT, j1 - jt);
    __syncthreads();
    for (int x = tid; x < cnt * D; x += BW_NT) tile[x] = q[(size_t)jt * D + x];
    __syncthreads();
    if (vi) {
      for (int j = 0; j < cnt; ++j) {
        float r2 = 0.f;
#pragma unroll
        for (int d = 0; d < D; ++d) {
          const float dd = xi[d] - tile[j * D + d];
          r2 = fmaf(dd, dd, r2);
        }
        const unsigned key = __float_as_uint(r2);
        if (pass == 0 || (key >> hi) == prefix) atomicAdd(&hist[(key >> shift) & mask], 1u);
      }
    }
  }
  __syncthreads();
  for (int b = tid; b < NBINS; b += BW_NT)
    if (hist[b]) atomicAdd(&ghist[b], (unsigned long long)hist[b]);
}

__global__ void k_sel_init(SelState *st, long long N, unsigned long long *ghist) {
  for (int b = threadIdx.x; b < NBINS; b += blockDim.x) ghist[b] = 0ull;
  if (threadIdx.x == 0) {
    const unsigned long long M = (unsigned long long)N * (unsigned long long)(N - 1) / 2ull;
    st->rank = (unsigned long long)N + 2ull * ((M - 1ull) / 2ull);
    st->prefix = 0u;
  }
}

__global__ void k_sel_digit(SelState *st, unsigned long long *ghist, int pass, long long N,
                            double *scal, int *err) {
  __shared__ int found;
  __shared__ unsigned long long below;
  if (threadIdx.x == 0) {
    const int nb = 1 << pass_bits(pass);
    unsigned long long cum = 0ull;
    found = -1;
    for (int b = 0; b < nb; ++b) {
      const unsigned long long c = ghist[b];
      if (st->rank < cum + c) {
        found = b;
        break;
      }
      cum += c;
    }
    below = cum;
  }
  __syncthreads();
  for (int b = threadIdx.x; b < NBINS; b += blockDim.x) ghist[b] = 0ull;
  if (threadIdx.x == 0) {
    if (found < 0) {
      vds_flag(err, VDS_ENAN);
      return;
    }
    st->rank -= below;
    st->prefix = (st->prefix << pass_bits(pass)) | (unsigned)found;
    if (pass == 2) {
      const float r2 = __uint_as_float(st->prefix);
      const double med = sqrt((double)r2);
      scal[SC_H] = med / sqrt(2.0 * log((double)N));
      scal[SC_AUX] = (double)r2;
      if (!(med > 0.0) || !(med < 1e300)) vds_flag(err, VDS_ENAN);
    }
  }
}

// ------------------------------------------------- bracketed selection

constexpr unsigned long long SMALL_PAIRS = 1ull << 22;
constexpr unsigned long long MOST_KEYS = 1ull << 30;  // 4 GiB of workspace: clouds of about three million particles
constexpr int SEL_NT = 512, SEL_BINS = 2048, SEL_BITS = 11;

// Selection of up to two order statistics among keys in [lo, hi], by digits of
// key - lo: what has been found so far (prefix) and the rank left inside it.
struct Sel {
  unsigned lo, hi;              // the bracket
  unsigned prefix[2], count[2];  // count: keys with the prefix
  unsigned long long rank[2];
  unsigned long long below;     // pairs with a key below lo
  unsigned long long in;        // pairs with a key in the bracket
  unsigned ticket, miss;
  // the screen: centre, largest |y|^2 (bits), and the widened bracket
  float mu[VDS_MAXD];
  unsigned ymax2;
  float slo, sspan;
};

__host__ __device__ __forceinline__ unsigned long long num_pairs(long long N) {
  return (unsigned long long)N * (unsigned long long)(N - 1) / 2ull;
}

__device__ __forceinline__ unsigned mix32(unsigned long long x) {  // splitmix64's finaliser
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return (unsigned)((x ^ (x >> 31)) >> 16);
}

template <int D>
__device__ __forceinline__ unsigned pair_key(const float *__restrict__ q, long i, long j) {
  float r2 = 0.f;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    const float dd = q[(size_t)i * D + d] - q[(size_t)j * D + d];
    r2 = fmaf(dd, dd, r2);
  }
  return __float_as_uint(r2);
}

// Keys of n pairs drawn with replacement (the draw depends on n alone).
template <int D>
__global__ void k_sample(const float *__restrict__ q, int N, long n, unsigned *__restrict__ keys) {
  for (long x = (long)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (long)gridDim.x * blockDim.x) {
    const long i = __umulhi(mix32(2 * x + 1), (unsigned)N);
    long j = __umulhi(mix32(2 * x + 2), (unsigned)(N - 1));
    j += j >= i;
    keys[x] = pair_key<D>(q, i, j);
  }
}

// All keys, pair (i < j) at i (2N - i - 1) / 2 + j - i - 1.
template <int D>
__global__ void k_all_keys(const float *__restrict__ q, int N, unsigned *__restrict__ keys) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= N) return;
  for (int i = blockIdx.y; i < j; i += gridDim.y)
    keys[(size_t)i * (2 * N - i - 1) / 2 + (j - i - 1)] = pair_key<D>(q, i, j);
}

__global__ void k_sel_start(Sel *s, unsigned *ghist, unsigned long long r0, unsigned long long r1) {
  for (int b = threadIdx.x; b < 2 * SEL_BINS; b += blockDim.x) ghist[b] = 0u;
  if (threadIdx.x == 0) {
    s->lo = 0u;
    s->hi = 0xffffffffu;
    s->prefix[0] = s->prefix[1] = 0u;
    s->rank[0] = r0;
    s->rank[1] = r1;
    s->below = s->in = 0ull;
    s->ticket = s->miss = 0u;
    s->ymax2 = 0u;
  }
}

// One digit of the selection of nt order statistics among `keys` (n of them,
// or s->in where n < 0): histograms of the keys that match what has been
// found, and the last CTA to finish picks the digits.  Level L takes the bits
// from shift(L) up; the levels cover 33 bits.
__device__ __forceinline__ int sel_shift(unsigned span, int level) {
  const int nb = 32 - __clz(span);
  const int s = nb - SEL_BITS * (level + 1);
  return s > 0 ? s : 0;
}

__global__ void __launch_bounds__(SEL_NT)
    k_sel_level(const unsigned *__restrict__ keys, long n_in, Sel *s, int level, int nt, unsigned *__restrict__ ghist) {
  __shared__ unsigned hist[2 * SEL_BINS];
  __shared__ unsigned long long wsum[SEL_NT / 32];
  __shared__ bool last;
  const int tid = threadIdx.x;
  const unsigned lo = s->lo, span = s->hi - lo;
  const int sh = sel_shift(span, level);
  const int up = level ? sel_shift(span, level - 1) : 32;
  if (s->miss || (level && up == 0)) return;  // nothing left to find
  const unsigned p0 = s->prefix[0], p1 = s->prefix[1];
  const long n = n_in >= 0 ? n_in : (long)s->in;
  for (int b = tid; b < nt * SEL_BINS; b += SEL_NT) hist[b] = 0u;
  __syncthreads();
  for (long x = (long)blockIdx.x * SEL_NT + tid; x < n; x += (long)gridDim.x * SEL_NT) {
    const unsigned v = keys[x] - lo;
    const unsigned pre = level ? v >> up : 0u;
    const unsigned dig = level ? (v >> sh) & ((1u << (up - sh)) - 1u) : v >> sh;
    if (pre == p0) atomicAdd(&hist[dig], 1u);
    if (nt > 1 && pre == p1) atomicAdd(&hist[SEL_BINS + dig], 1u);
  }
  __syncthreads();
  for (int b = tid; b < nt * SEL_BINS; b += SEL_NT)
    if (hist[b]) atomicAdd(&ghist[b], hist[b]);
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(&s->ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  constexpr int PT = SEL_BINS / SEL_NT;  // bins per thread
  for (int t = 0; t < nt; ++t) {
    const unsigned long long rank = s->rank[t];
    unsigned long long c[PT], sum = 0ull;
#pragma unroll
    for (int k = 0; k < PT; ++k) {
      c[k] = __ldcg(&ghist[t * SEL_BINS + tid * PT + k]);
      sum += c[k];
    }
    // exclusive prefix sum over the threads
    unsigned long long inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, inc, o);
      if ((tid & 31) >= o) inc += y;
    }
    if ((tid & 31) == 31) wsum[tid >> 5] = inc;
    __syncthreads();
    unsigned long long base = inc - sum;
    for (int w = 0; w < (tid >> 5); ++w) base += wsum[w];
    __syncthreads();
    if (rank >= base && rank < base + sum) {  // one thread at most
#pragma unroll
      for (int k = 0; k < PT; ++k) {
        if (rank >= base && rank < base + c[k]) {
          s->rank[t] = rank - base;
          s->count[t] = (unsigned)c[k];
          s->prefix[t] = level ? (s->prefix[t] << (up - sh)) | (unsigned)(tid * PT + k) : (unsigned)(tid * PT + k);
        }
        base += c[k];
      }
    }
  }
  for (int b = tid; b < nt * SEL_BINS; b += SEL_NT) ghist[b] = 0u;
  if (tid == 0) s->ticket = 0u;
}

// Screen records: y = x - mu and |y|^2, padded to four floats.
template <int D>
struct Scr {
  static constexpr int DP = (D + 1 + 3) / 4 * 4;
};

// mu = the mean of up to 4096 particles (any centre is right; a central one
// keeps the bound small).  One CTA.
template <int D>
__global__ void __launch_bounds__(512) k_centre(const float *__restrict__ q, int N, Sel *s) {
  __shared__ float sh[16][D];
  const int n = min(N, 4096), stride = N / n, tid = threadIdx.x;
  float m[D];
#pragma unroll
  for (int d = 0; d < D; ++d) m[d] = 0.f;
  for (int x = tid; x < n; x += 512)
#pragma unroll
    for (int d = 0; d < D; ++d) m[d] += q[(size_t)x * stride * D + d];
#pragma unroll
  for (int d = 0; d < D; ++d) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m[d] += __shfl_xor_sync(0xffffffffu, m[d], o);
    if ((tid & 31) == 0) sh[tid >> 5][d] = m[d];
  }
  __syncthreads();
  if (tid < D) {
    float v = 0.f;
    for (int w = 0; w < 16; ++w) v += sh[w][tid];
    s->mu[tid] = v / (float)n;
  }
}

template <int D>
__global__ void k_screen_rec(const float *__restrict__ q, int N, Sel *s, float *__restrict__ rec) {
  constexpr int DP = Scr<D>::DP;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  float n2 = 0.f;
  if (i < N) {
    float o[DP];
#pragma unroll
    for (int d = 0; d < DP; ++d) o[d] = 0.f;
#pragma unroll
    for (int d = 0; d < D; ++d) {
      o[d] = q[(size_t)i * D + d] - s->mu[d];
      n2 = fmaf(o[d], o[d], n2);
    }
    o[D] = n2;
#pragma unroll
    for (int v = 0; v < DP / 4; ++v)
      reinterpret_cast<float4 *>(rec + (size_t)i * DP)[v] =
          make_float4(o[4 * v], o[4 * v + 1], o[4 * v + 2], o[4 * v + 3]);
  }
  // NaN and infinity have the largest patterns
  const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(n2) & 0x7fffffffu);
  if ((threadIdx.x & 31) == 0) atomicMax(&s->ymax2, m);
}

// The bracket from the two prefixes that `levels` levels of a 32-bit span found in
// the sample of n keys (order statistics r0 and r1), the state of the pass that
// uses it, and the screen's.  With u = 2^-24 and Y^2 >= |y|^2 for every particle,
// the screen value differs from the key's float (both of the pair's true squared
// distance) by at most
//   2D u Y^2 (the norms) + 5 u Y^2 (|y_i|^2 - slo) + 6 u Y^2 (their sum) +
//   8D u Y^2 (D fused steps of partial sums up to 8 Y^2) + 8 u Y^2 (rounding
//   y) + 4 (D + 2) u Y^2 (the key)  =  (14D + 27) u Y^2.
// A miss at once where the sample says that the bracket holds more keys than
// there is room for (equal distances), or that the widened one holds over 2 % of
// the pairs, as the queue of the pass then takes longer than the histograms save.
__global__ void k_sel_bracket(Sel *s, int D, int levels, unsigned long long r0, unsigned long long r1,
                              unsigned long long n, unsigned long long M, unsigned long long cap) {
  const int sh = sel_shift(0xffffffffu, levels - 1);
  s->lo = s->prefix[0] << sh;
  s->hi = (s->prefix[1] << sh) | ((1u << sh) - 1u);
  s->prefix[0] = 0u;
  const double lo = __uint_as_float(s->lo), hi = __uint_as_float(s->hi), y2 = __uint_as_float(s->ymax2);
  const double eps = (14.0 * D + 40.0) * 5.9604644775390625e-8 * y2 * 1.0001;
  // part of the sample, and so of the pairs, inside
  const double in = (double)((r1 - s->rank[1] + s->count[1]) - (r0 - s->rank[0])) / (double)n;
  const double width = hi > lo ? hi - lo : 0.0;
  if (!(y2 < 1e30 && hi < 1e30 && in * (double)M <= 0.99 * (double)cap && in * (width + 2.0 * eps) <= 0.02 * width))
    s->miss = 1u;
  s->slo = __double2float_rd(lo - eps);
  s->sspan = __double2float_ru((hi + eps) - (double)s->slo);
}

// The selection among the collected keys starts where the median lies in the
// bracket: rank minus the pairs below; a miss where it does not.
__global__ void k_sel_collected(Sel *s, unsigned long long rank, unsigned long long cap) {
  if (s->miss || rank < s->below || rank >= s->below + s->in || s->in > cap) s->miss = 1u;
  else s->rank[0] = rank - s->below;
}

__global__ void k_sel_done(const Sel *s, long long N, double *scal) {
  const float r2 = __uint_as_float(s->lo + s->prefix[0]);
  const double med = sqrt((double)r2);
  scal[SC_H] = med / sqrt(2.0 * log((double)N));
  scal[SC_AUX] = (double)r2;
  // what the host acts on: not finite or zero, or another path is needed
  scal[SC_AUX + 1] = s->miss ? 2.0 : (!(med > 0.0) || !(med < 1e300)) ? 1.0 : 0.0;
}

// Shapes of the pass over all pairs: particles per thread in registers, one
// record at a time from shared memory (broadcast).
template <int D>
struct BrCfg {
  static constexpr int NT = 128, RI = D <= 10 ? 8 : 4, TI = NT * RI, TJ = 64;
  static constexpr int DP = Scr<D>::DP;
  static constexpr int MINB = 4;
};
constexpr int BR_QUEUE = 1024;

// Over the unordered pairs of sc's triangle of (i-tile, j-chunk) items: keys
// below lo counted, keys in [lo, hi] written to keys[0, cap) (in any order:
// what follows is a selection).  s->in counts all of them, also those past cap.
template <int D>
__global__ void __launch_bounds__(BrCfg<D>::NT, BrCfg<D>::MINB)
    k_bracket(const float *__restrict__ q, const float *__restrict__ rec, int N, Sched sc, Sel *s,
              unsigned *__restrict__ keys, unsigned long long cap) {
  using C = BrCfg<D>;
  constexpr int NT = C::NT, RI = C::RI, TJB = C::TJ, DP = C::DP, CPT = C::TI / TJB;
  static_assert(TJB <= 256 && RI <= 8, "queue entries: thread, eight bits of j, a bit for each of its particles");
  __shared__ __align__(16) float tile[2][TJB * DP];
  __shared__ unsigned queue[BR_QUEUE], kept[2 * BR_QUEUE];
  __shared__ unsigned qn, kn;
  __shared__ unsigned long long kbase;
  const int tid = threadIdx.x, lane = tid & 31;
  const long long it0 = (long long)blockIdx.x * sc.items / sc.G;
  const long long it1 = (long long)(blockIdx.x + 1) * sc.items / sc.G;
  if (it0 >= it1 || s->miss) return;
  const unsigned lo = s->lo, span = s->hi - lo;
  const float slo = s->slo;
  const unsigned sspan = __float_as_uint(s->sspan);
  int t = 0;
  {
    int a = 0, b = sc.n_itiles;
    while (b - a > 1) {
      const int m = (a + b) >> 1;
      if (sched_start(m, sc) <= it0) a = m;
      else b = m;
    }
    t = a;
  }
  int c = t * CPT + (int)(it0 - sched_start(t, sc));
  auto stage = [&](int chunk, int buf) {
    const int n = min(TJB, N - chunk * TJB);
    const float *src = rec + (size_t)chunk * TJB * DP;
    for (int x = tid; x < n * (DP / 4); x += NT) cp_async16(&tile[buf][4 * x], src + 4 * x);
  };
  unsigned long long total = 0ull;
  // a pair of the screen's bracket: its key decides
  auto sort_in = [&](unsigned key, bool on) {
    total += on && key < lo;
    const bool in = on && key - lo <= span;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if (m == 0u) return;
    unsigned base = 0u;
    if (lane == 0) base = atomicAdd(&kn, (unsigned)__popc(m));
    base = __shfl_sync(0xffffffffu, base, 0) + __popc(m & ((1u << lane) - 1u));
    if (in) {
      if (base < 2 * BR_QUEUE) {
        kept[base] = key;
      } else {
        const unsigned long long p = atomicAdd(&s->in, 1ull);
        if (p < cap) keys[p] = key;
      }
    }
  };
  auto flush = [&]() {  // all threads; kept[] is complete
    const unsigned m = min(kn, 2u * BR_QUEUE);
    if (tid == 0 && m) kbase = atomicAdd(&s->in, (unsigned long long)m);
    __syncthreads();
    for (unsigned x = tid; x < m; x += NT)
      if (kbase + x < cap) keys[kbase + x] = kept[x];
    __syncthreads();
    if (tid == 0) kn = 0u;
  };
  stage(c, 0);
  if (tid == 0) qn = kn = 0u;
  float xi[RI][D], ni[RI];
  int cur = -1;
  cp_async_wait_all();
  __syncthreads();
  for (long long it = it0; it < it1; ++it) {
    const int b = (int)((it - it0) & 1);
    if (t != cur) {
      cur = t;
#pragma unroll
      for (int k = 0; k < RI; ++k) {
        const int i = min(t * C::TI + tid + k * NT, N - 1);
#pragma unroll
        for (int d = 0; d < D; ++d) xi[k][d] = -2.f * rec[(size_t)i * DP + d];
        ni[k] = rec[(size_t)i * DP + D] - slo;
      }
    }
    int tn = t, cn = c + 1;
    if (cn == sc.nchunk) {
      ++tn;
      cn = tn * CPT;
    }
    if (it + 1 < it1) stage(cn, b ^ 1);
    const float *tl = tile[b];
    const int cnt = min(TJB, N - c * TJB);
    unsigned below = 0u;
    auto load = [&](int j, float (&xj)[DP]) {
#pragma unroll
      for (int v = 0; v < DP / 4; ++v) {
        const float4 f = reinterpret_cast<const float4 *>(tl + j * DP)[v];
        xj[4 * v] = f.x;
        xj[4 * v + 1] = f.y;
        xj[4 * v + 2] = f.z;
        xj[4 * v + 3] = f.w;
      }
    };
    auto pass = [&](auto own) {  // own: the tile's own chunks, pairs i < j only
      for (int j = 0; j < cnt; ++j) {
        float xj[DP];
        load(j, xj);
        unsigned v[RI], least = 0xffffffffu;
#pragma unroll
        for (int k = 0; k < RI; ++k) {
          float r = ni[k] + xj[D];
#pragma unroll
          for (int d = 0; d < D; ++d) r = fmaf(xi[k][d], xj[d], r);
          v[k] = __float_as_uint(r);  // screen value minus slo: the sign bit says below
          if (own && t * C::TI + tid + k * NT >= c * TJB + j) v[k] = 0x7fffffffu;
          below += v[k] >> 31;
          least = min(least, v[k]);
        }
        if (least <= sspan) {  // one queue entry for the thread's pairs with this j
          unsigned hits = 0u;
#pragma unroll
          for (int k = 0; k < RI; ++k) hits |= v[k] <= sspan ? 1u << k : 0u;
          const unsigned pos = atomicAdd(&qn, 1u);
          if (pos < BR_QUEUE) queue[pos] = (unsigned)tid << 16 | (unsigned)j << 8 | hits;
          else
            for (; hits; hits &= hits - 1u) {
              const unsigned key = pair_key<D>(q, t * C::TI + tid + (__ffs(hits) - 1) * NT, c * TJB + j);
              total += key < lo;
              if (key - lo <= span) {
                const unsigned long long p = atomicAdd(&s->in, 1ull);
                if (p < cap) keys[p] = key;
              }
            }
        }
      }
    };
    if (c >= (t + 1) * CPT) pass(std::false_type{});  // every j after every i of the tile
    else pass(std::true_type{});
    total += below;
    cp_async_wait_all();
    __syncthreads();
    const unsigned held = min(qn, (unsigned)BR_QUEUE);
    for (unsigned x0 = 0; x0 < held; x0 += NT) {
      unsigned w = x0 + tid < held ? queue[x0 + tid] : 0u;
      while (__any_sync(0xffffffffu, w & 0xffu)) {  // nearly always one pair per entry
        const bool on = (w & 0xffu) != 0u;
        const int i = t * C::TI + (int)(w >> 16) + (__ffs(w & 0xffu) - 1) * NT;
        sort_in(on ? pair_key<D>(q, i, c * TJB + (int)(w >> 8 & 0xffu)) : 0u, on);
        w &= w - 1u;
        if (!on) w = 0u;
      }
    }
    __syncthreads();
    if (tid == 0) qn = 0u;
    if (kn >= BR_QUEUE) flush();  // kn is settled: uniform
    __syncthreads();
    t = tn;
    c = cn;
  }
  flush();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
  if (lane == 0 && total) atomicAdd(&s->below, total);
}

// The bracketed selection; done = false where it has to be taken over by the
// histograms (a miss, or no memory for the keys).  Synchronises.
template <int D>
int select_impl(vds_ctx *c, const float *q, int N, bool &done) {
  done = false;
  const unsigned long long M = num_pairs(N), rank = (M - 1ull) / 2ull;
  const bool small = M <= SMALL_PAIRS;
  // sample: from (7.5 M)^(2/3) on (N above 350000) it would hold more keys than
  // the bracket it gives
  unsigned long long n = M / 1024;
  if (n > (1ull << 20)) n = (unsigned long long)fmin((double)n, cbrt(7.5 * (double)M) * cbrt(7.5 * (double)M));
  if (n < (1ull << 20)) n = 1ull << 20;
  const double half = 2.5 * sqrt((double)n);
  // room for the sample, then for half as many keys again as the bracket holds on average
  const unsigned long long want = small ? M : (unsigned long long)(1.5 * 2.0 * half / (double)n * (double)M);
  const unsigned long long cap = small ? M : (want > n ? want : n);
  VDS_TRY(vds_ensure(c, c->red, sizeof(Sel) + 2 * SEL_BINS * sizeof(unsigned)));
  int st = cap <= MOST_KEYS ? vds_ensure_spare(c, c->part, cap * sizeof(unsigned)) : VDS_ENOMEM;
  if (st == VDS_OK && !small) st = vds_ensure(c, c->rec, (size_t)N * Scr<D>::DP * sizeof(float));
  if (st == VDS_ENOMEM) {
    (void)cudaGetLastError();
    return VDS_OK;
  }
  VDS_TRY(st);
  Sel *s = (Sel *)c->red.ptr;
  unsigned *gh = (unsigned *)((char *)c->red.ptr + sizeof(Sel)), *keys = (unsigned *)c->part.ptr;
  auto level = [&](long cnt, unsigned long long expect, int l, int nt) {
    unsigned long long g = (expect + SEL_NT * 8 - 1) / (SEL_NT * 8);
    const unsigned long long most = 2ull * c->num_sms;
    k_sel_level<<<(unsigned)(g < 1 ? 1 : g > most ? most : g), SEL_NT, 0, c->stream>>>(keys, cnt, s, l, nt, gh);
    ++c->launches;
  };
  if (small) {
    k_sel_start<<<1, 512, 0, c->stream>>>(s, gh, rank, 0ull);
    VDS_TRY(vds_time_begin(c, PK_BANDWIDTH));
    const int bx = (N + 127) / 128;
    k_all_keys<D><<<dim3(bx, (8 * c->num_sms + bx - 1) / bx), 128, 0, c->stream>>>(q, N, keys);
    VDS_TRY(vds_time_end(c, PK_BANDWIDTH));
    for (int l = 0; l < 3; ++l) level((long)M, M, l, 1);
    c->launches += 2;
  } else {
    const unsigned long long r0 = (unsigned long long)(0.5 * (double)n - half),
                             r1 = (unsigned long long)(0.5 * (double)n + half);
    // the top 22 bits of the keys resolve the bracket of a small sample
    const int levels = n > (1ull << 23) ? 3 : 2;
    k_sel_start<<<1, 512, 0, c->stream>>>(s, gh, r0, r1);
    k_sample<D><<<8 * c->num_sms, 256, 0, c->stream>>>(q, N, (long)n, keys);
    for (int l = 0; l < levels; ++l) level((long)n, n, l, 2);
    k_centre<D><<<1, 512, 0, c->stream>>>(q, N, s);
    float *rec = (float *)c->rec.ptr;
    k_screen_rec<D><<<(N + 255) / 256, 256, 0, c->stream>>>(q, N, s, rec);
    k_sel_bracket<<<1, 1, 0, c->stream>>>(s, D, levels, r0, r1, n, M, cap);
    using C = BrCfg<D>;
    Sched sc;
    sc.TI = C::TI;
    sc.nchunk = (N + C::TJ - 1) / C::TJ;
    sc.cpt = C::TI / C::TJ;
    sc.n_itiles = (N + C::TI - 1) / C::TI;
    sc.items = sched_start(sc.n_itiles, sc);
    sc.Npad = sc.Nipad = N;
    sc.maxseg = 0;
    const long long g = (long long)c->num_sms * C::MINB;
    sc.G = (int)(sc.items < g ? sc.items : g);
    VDS_TRY(vds_time_begin(c, PK_BANDWIDTH));
    k_bracket<D><<<sc.G, C::NT, 0, c->stream>>>(q, rec, N, sc, s, keys, cap);
    VDS_TRY(vds_time_end(c, PK_BANDWIDTH));
    k_sel_collected<<<1, 1, 0, c->stream>>>(s, rank, cap);
    for (int l = 0; l < 3; ++l) level(-1, (unsigned long long)(2.0 * half / (double)n * (double)M), l, 1);
    c->launches += 5 + levels;
  }
  k_sel_done<<<1, 1, 0, c->stream>>>(s, N, c->scal);
  ++c->launches;
  VDS_CUDA_TRY(cudaGetLastError());
  VDS_CUDA_TRY(cudaMemcpyAsync(c->h_scal, c->scal, SC_COUNT * sizeof(double), cudaMemcpyDeviceToHost,
                               c->stream));
  VDS_TRY(vds_sync_status(c));
  const double what = c->h_scal[SC_AUX + 1];
  if (what == 2.0) return VDS_OK;
  done = true;
  return what == 0.0 ? VDS_OK : VDS_ENAN;
}

// Silverman: per-coordinate FP64 mean, then sum of squared deviations.
template <int D>
__global__ void __launch_bounds__(256)
    k_moments(const float *__restrict__ q, int N, int pass, double *red, unsigned *ticket,
              double *scal) {
  __shared__ double sh[8][D];
  __shared__ bool last;
  double acc[D];
#pragma unroll
  for (int d = 0; d < D; ++d) acc[d] = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
#pragma unroll
    for (int d = 0; d < D; ++d) {
      const double v = (double)q[(size_t)i * D + d];
      if (pass == 0) acc[d] += v;
      else {
        const double x = v - scal[SC_AUX + d];
        acc[d] += x * x;
      }
    }
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int d = 0; d < D; ++d) {
    double v = acc[d];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) sh[w][d] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int d = 0; d < D; ++d) {
      double v = 0.0;
      for (int k = 0; k < (int)(blockDim.x >> 5); ++k) v += sh[k][d];
      red[(size_t)blockIdx.x * D + d] = v;
    }
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last || threadIdx.x != 0) return;
  __threadfence();
  double sig = 0.0;
  for (int d = 0; d < D; ++d) {
    double v = 0.0;
    for (unsigned b = 0; b < gridDim.x; ++b) v += __ldcg(red + (size_t)b * D + d);
    if (pass == 0) scal[SC_AUX + d] = v / (double)N;
    else sig += sqrt(v / (double)(N - 1));
  }
  if (pass == 1) {
    sig /= (double)D;
    scal[SC_H] = sig * pow(4.0 / ((double)(D + 2) * (double)N), 1.0 / (double)(D + 4));
  }
  *ticket = 0u;
}

template <int D>
int bandwidth_impl(vds_ctx *c, const float *q, int N, int rule, double *h) {
  if (rule == 1) {
    int nblk = (N + 255) / 256;
    if (nblk > 2 * c->num_sms) nblk = 2 * c->num_sms;
    VDS_TRY(vds_ensure(c, c->red, (size_t)nblk * D * sizeof(double)));
    for (int pass = 0; pass < 2; ++pass) {
      k_moments<D><<<nblk, 256, 0, c->stream>>>(q, N, pass, (double *)c->red.ptr, c->ticket + TK_MISC,
                                                c->scal);
      VDS_CUDA_TRY(cudaGetLastError());
      ++c->launches;
    }
  } else {
    bool done = false;
    VDS_TRY(select_impl<D>(c, q, N, done));
    if (done) {
      *h = c->h_scal[SC_H];
      return VDS_OK;
    }
    // state + global histogram live in the reduction scratch
    VDS_TRY(vds_ensure(c, c->red, sizeof(SelState) + NBINS * sizeof(unsigned long long)));
    SelState *st = (SelState *)c->red.ptr;
    unsigned long long *gh = (unsigned long long *)((char *)c->red.ptr + sizeof(SelState));
    k_sel_init<<<1, 256, 0, c->stream>>>(st, N, gh);
    VDS_CUDA_TRY(cudaGetLastError());
    ++c->launches;
    const int n_itiles = (N + BW_NT - 1) / BW_NT;
    // split j so that the grid covers the GPU a few times over
    int nsplit = (4 * c->num_sms + n_itiles - 1) / n_itiles;
    if (nsplit < 1) nsplit = 1;
    int jchunk = (N + nsplit - 1) / nsplit;
    jchunk = (jchunk + BW_NT - 1) / BW_NT * BW_NT;
    nsplit = (N + jchunk - 1) / jchunk;
    for (int pass = 0; pass < 3; ++pass) {
      VDS_TRY(vds_time_begin(c, PK_BANDWIDTH));
      k_hist<D><<<dim3(n_itiles, nsplit), BW_NT, 0, c->stream>>>(q, N, jchunk, st, pass, gh);
      VDS_CUDA_TRY(cudaGetLastError());
      VDS_TRY(vds_time_end(c, PK_BANDWIDTH));
      ++c->launches;
      k_sel_digit<<<1, 256, 0, c->stream>>>(st, gh, pass, N, c->scal, c->err);
      VDS_CUDA_TRY(cudaGetLastError());
      ++c->launches;
    }
  }
  VDS_CUDA_TRY(cudaMemcpyAsync(c->h_scal, c->scal, SC_COUNT * sizeof(double), cudaMemcpyDeviceToHost,
                               c->stream));
  VDS_TRY(vds_sync_status(c));
  *h = c->h_scal[SC_H];
  return VDS_OK;
}

}  // namespace

extern "C" int vds_bandwidth(vds_ctx *c, const float *q, int N, int D, int rule, double *h) {
  if (!c || !q || !h || N < 2 || (rule != 0 && rule != 1)) return VDS_EARG;
  int prev = -1;
  cudaGetDevice(&prev);
  if (prev != c->device) cudaSetDevice(c->device);
  int st;
  switch (D) {
    case 2: st = bandwidth_impl<2>(c, q, N, rule, h); break;
    case 3: st = bandwidth_impl<3>(c, q, N, rule, h); break;
    case 4: st = bandwidth_impl<4>(c, q, N, rule, h); break;
    case 6: st = bandwidth_impl<6>(c, q, N, rule, h); break;
    case 8: st = bandwidth_impl<8>(c, q, N, rule, h); break;
    case 9: st = bandwidth_impl<9>(c, q, N, rule, h); break;
    case 10: st = bandwidth_impl<10>(c, q, N, rule, h); break;
    case 12: st = bandwidth_impl<12>(c, q, N, rule, h); break;
    case 14: st = bandwidth_impl<14>(c, q, N, rule, h); break;
    case 15: st = bandwidth_impl<15>(c, q, N, rule, h); break;
    case 16: st = bandwidth_impl<16>(c, q, N, rule, h); break;
    default: st = VDS_EARG;
  }
  if (prev >= 0 && prev != c->device) cudaSetDevice(prev);
  return st;
}
