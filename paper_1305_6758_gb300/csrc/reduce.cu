// Cross-path reduction: per-path records -> ensemble estimates (FP64
// throughout), the covariance backward, and a Philox kernel for stream checks.
//
// Estimates follow Sec. 2.2 of Rakic et al.: the MC average over paths,
// Eq. (MCAV); chi and C_V from the fluctuation formulas, Eq. (cv); the Binder
// cumulant, Eq. (kum); the coefficient of variation of a mean, Eq. (eq:cv);
// and the distribution coefficient of the normal Q-Q line fit, Eq.
// (dist-coefficient) of Sec. 3.  Standard errors of derived quantities are
// delete-one jackknife over paths (paths are independent, so no blocking).
//
// What bounds it is FP64 issue (76 cycles per warp instruction and scheduler
// on GB300), so it is spread over the SMs and does each FP64 step once: up to
// 32 CTAs of 128 threads per system (one warp per scheduler) sum the fields,
// then a second pass takes variances and jackknife together; the normal
// quantiles are evaluated once for half the paths (they are antisymmetric)
// instead of twelve times for all of them; the six sorts run in CTAs of
// their own on integer keys.  Against one CTA per system: 4096 paths x 21
// systems 1.93 -> 0.14 ms, 10^4 paths x 4 5.5 -> 0.22 ms, 256 paths 0.40 -> 0.044 ms,
// 90112 paths 84 -> 1.7 ms.
#include <cmath>
#include <cstdint>

#include "common.cuh"
#include "kernels.h"
#include "philox.cuh"

namespace mpk {

static_assert(sizeof(mp_estimates_t) == MP_NEST * sizeof(double), "estimates layout");

constexpr int kBackThreads = 512;  // backward
constexpr int kRedThreads = 128;   // one warp per scheduler: FP64 issue is what the passes wait for
constexpr int kRedMaxCtas = 32;    // CTAs per system (their partial sums are added one by one)
constexpr int kSortThreads = 1024;
constexpr int kNumMean = 13;  // record fields MP_R_E .. MP_R_MMZ
constexpr int kNumDerived = 9;
constexpr int kNumR = 6;      // fields with a distribution coefficient
__constant__ const int kRField[kNumR] = {MP_R_E, MP_R_M, MP_R_MX, MP_R_MY, MP_R_MZ, MP_R_AMZ};

// Scratch of one system (doubles, from ReduceParams::work + rec_offset + 64 system):
// [partial sums: nb x kRedPart][S_xq: 6 x nb, S_xq of large systems][counter][quantiles: ceil(P/2)]
// with nb = reduce_ctas(P) <= P/128 + 1, together at most P + 64.
constexpr int kSums = kNumMean + 1 + 4 + 2;                    // fields, acceptance, half sums, S_qq, worst norm
constexpr int kVars = kNumMean + 1 + 4 + 2 * kNumDerived;      // variances, half variances, jackknife sums
constexpr int kRedPart = kSums + kVars + kNumR;
__host__ __device__ inline int reduce_ctas(int64_t P) {
  const int64_t n = (P + kRedThreads - 1) / kRedThreads;
  return n < kRedMaxCtas ? static_cast<int>(n) : kRedMaxCtas;
}
static_assert(kRedPart <= 62, "scratch of one system: 62 (P/128 + 1) + 1 + (P+1)/2 <= P + 64");

struct ReduceScratch {
  double *sums, *vars, *xq, *q;
  unsigned* done;
  __device__ ReduceScratch(const ReduceParams& p, int sidx, int64_t rec_offset, int64_t P) {
    const int nb = reduce_ctas(P);
    sums = p.work + rec_offset + 64 * static_cast<int64_t>(sidx);
    vars = sums + nb * kSums;
    xq = vars + nb * kVars;
    done = reinterpret_cast<unsigned*>(xq + nb * kNumR);
    q = xq + nb * kNumR + 1;
  }
};

// Sum V values over the CTA; every thread receives the totals.
template <int V>
__device__ void block_sum(double (&v)[V], double* scratch) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int k = 0; k < V; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < V; ++k) scratch[warp * V + k] = v[k];
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < V; ++k) {
    double t = 0.0;
    for (int w = 0; w < nw; ++w) t += scratch[w * V + k];
    v[k] = t;
  }
  __syncthreads();
}

// The totals of V values over a CTA of kRedThreads threads, in total[0..V).
// Every lane of the FP64 pipe counts: the values go through shared memory and
// thread (value, part) adds one part of the rows, kRedThreads V / 32 adds
// issued over the CTA instead of the 5 V per warp of a butterfly (36 values:
// 3.5 us instead of 12).
template <int V>
struct TotalBuf {
  static constexpr int kRow = V | 1;  // odd: a warp's rows fall on different banks
  static constexpr int kParts = kRedThreads / V;
  double rows[kRedThreads * kRow], part[kParts * V], total[V];
};
template <int V>
__device__ void block_total(const double (&v)[V], TotalBuf<V>& b) {
  constexpr int kParts = TotalBuf<V>::kParts, kRow = TotalBuf<V>::kRow;
  const int tid = threadIdx.x, k = tid % V, part = tid / V;
#pragma unroll
  for (int j = 0; j < V; ++j) b.rows[tid * kRow + j] = v[j];
  __syncthreads();
  if (part < kParts) {
    double t = 0.0;
    for (int r = part; r < kRedThreads; r += kParts) t += b.rows[r * kRow + k];
    b.part[part * V + k] = t;
  }
  __syncthreads();
  if (tid < V) {
    double t = b.part[tid];
    for (int q = 1; q < kParts; ++q) t += b.part[q * V + tid];
    b.total[tid] = t;
  }
  __syncthreads();
}

// chi, C_V, U_L and the six fluctuation derivatives from pooled means
// (indexed by MP_R_*).  Under the weight exp(-beta N e):
//   d<A>/dbeta = -N cov(A, e),   d<A>/dh = <dA/dh> + beta N cov(A, m_z),
// and of A in {e, |m|, m_z} only e = (-J E_bonds - h M_z)/N depends on h
// itself (de/dh = -m_z).
__device__ void derived(const double* mu, double N, double beta, double* th) {
  const double e = mu[MP_R_E], e2 = mu[MP_R_E2], m = mu[MP_R_M], m2 = mu[MP_R_M2];
  const double m4 = mu[MP_R_M4], mz = mu[MP_R_MZ], mz2 = mu[MP_R_MZ2];
  const double em = mu[MP_R_EM], emz = mu[MP_R_EMZ], mmz = mu[MP_R_MMZ];
  th[0] = N * beta * (m2 - m * m);          // chi
  th[1] = N * beta * beta * (e2 - e * e);   // C_V
  th[2] = 1.0 - m4 / (3.0 * m2 * m2);       // Binder U_L
  th[3] = -N * (e2 - e * e);                // d<e>/dbeta
  th[4] = -N * (em - m * e);                // d<|m|>/dbeta
  th[5] = -N * (emz - mz * e);              // d<m_z>/dbeta
  th[6] = beta * N * (emz - e * mz) - mz;   // d<e>/dh: e's own field term adds -<m_z>
  th[7] = beta * N * (mmz - m * mz);        // d<|m|>/dh
  th[8] = beta * N * (mz2 - mz * mz);       // d<m_z>/dh
}

// Pass 1: sums of the record fields, of e and |m| over each half of the paths
// (Sec. 4's two-start check: paths 0 .. Pa-1 and Pa .. P-1, Pa = ceil(P/2)),
// the worst norm, and the normal quantiles at (i + 1/2)/P, i < P/2 (the
// others are their negatives; an odd P's middle one is 0).
__global__ void __launch_bounds__(kRedThreads) reduce_sums_kernel(const ReduceParams p) {
  __shared__ TotalBuf<kSums> buf;
  const int sidx = blockIdx.y;
  const DevSystem& sy = p.systems[sidx];
  const int64_t P = sy.n_paths;
  const int nb = reduce_ctas(P);
  if (static_cast<int>(blockIdx.x) >= nb) return;
  const ReduceScratch w(p, sidx, sy.rec_offset, P);
  if (blockIdx.x == 0 && threadIdx.x == 0) *w.done = 0u;
  const double* rec = p.records + sy.rec_offset * MP_NREC;
  const int64_t Pa = P - P / 2, half = P / 2;
  const int64_t first = static_cast<int64_t>(blockIdx.x) * kRedThreads + threadIdx.x, step = nb * kRedThreads;
  double v[kSums];
#pragma unroll
  for (int k = 0; k < kSums; ++k) v[k] = 0.0;
  double worst = 0.0;
  for (int64_t i = first; i < P; i += step) {
    const double* r = rec + i * MP_NREC;
#pragma unroll
    for (int k = 0; k < kNumMean; ++k) {
      if (k != MP_R_E && k != MP_R_M) v[k] += r[k];
    }
    const int a = i < Pa ? 0 : 1;
    const double e = r[MP_R_E], m = r[MP_R_M];
    v[kNumMean + 1] += a ? 0.0 : e;
    v[kNumMean + 2] += a ? 0.0 : m;
    v[kNumMean + 3] += a ? e : 0.0;
    v[kNumMean + 4] += a ? m : 0.0;
    v[kNumMean] += r[MP_R_ACC];
    worst = fmax(worst, r[MP_R_NORM]);
  }
  const double invP = 1.0 / static_cast<double>(P);
  for (int64_t i = first; i < half; i += step) {
    const double q = normcdfinv((i + 0.5) * invP);
    w.q[i] = q;
    v[kSums - 2] += 2.0 * q * q;
  }
  v[MP_R_E] = v[kNumMean + 1] + v[kNumMean + 3];
  v[MP_R_M] = v[kNumMean + 2] + v[kNumMean + 4];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) worst = fmax(worst, __shfl_xor_sync(0xffffffffu, worst, o));
  __shared__ double wmax[kRedThreads / 32];
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = worst;
  block_total<kSums>(v, buf);
  if (threadIdx.x < kSums) {
    double t = buf.total[threadIdx.x];
    if (threadIdx.x == kSums - 1)
      for (int k = 0; k < kRedThreads / 32; ++k) t = fmax(t, wmax[k]);
    w.sums[blockIdx.x * kSums + threadIdx.x] = t;
  }
}

// Doubles as integers of the same order (the sort compares on the integer
// pipes, not the FP64 one).
__device__ __forceinline__ int64_t order_key(double x) {
  const int64_t b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double key_value(int64_t k) {
  return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll));
}

// Bitonic stages of size k with strides j0, j0/2, ..., 1 on the n keys of
// shared memory whose first element has index `base` in the whole array.
__device__ void bitonic_strides(int64_t* keys, int n, int64_t base, int64_t k, int j0) {
  for (int j = j0; j > 0; j >>= 1) {
    for (int t = threadIdx.x; t < n / 2; t += blockDim.x) {
      const int i = 2 * t - (t & (j - 1));  // the pair (i, i + j)
      const int64_t a = keys[i], b = keys[i + j];
      if ((a > b) == (((base + i) & k) == 0)) {
        keys[i] = b;
        keys[i + j] = a;
      }
    }
    __syncthreads();
  }
}

__device__ inline int64_t pow2_above(int64_t P) {
  int64_t n = 1;
  while (n < P) n <<= 1;
  return n;
}

// Eq. (dist-coefficient) of one record field: with the sorted values fitted
// to the normal quantiles by least squares, r = 1 - SS_res / ((P-1) sigma^2)
// = S_xq^2 / (S_xx S_qq).  S_xx is the field's variance sum, and since the
// quantiles are antisymmetric S_xq = sum_{i < P/2} q_i (x_(i) - x_(P-1-i)).
// One CTA sorts one field of one system in shared memory.
__global__ void __launch_bounds__(kSortThreads) reduce_sort_kernel(const ReduceParams p) {
  extern __shared__ __align__(16) int64_t keys[];
  __shared__ double scratch[kSortThreads / 32];
  const int sidx = blockIdx.y, f = blockIdx.x;
  const DevSystem& sy = p.systems[sidx];
  const int64_t P = sy.n_paths;
  if (P < 3 || P > MP_R_MAX_PATHS) return;
  const ReduceScratch w(p, sidx, sy.rec_offset, P);
  const double* x = p.records + sy.rec_offset * MP_NREC + kRField[f];
  const int n = static_cast<int>(pow2_above(P));
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    keys[i] = order_key(i < P ? x[static_cast<int64_t>(i) * MP_NREC] : INFINITY);
  __syncthreads();
  for (int k = 2; k <= n; k <<= 1) bitonic_strides(keys, n, 0, k, k >> 1);
  double s[1] = {0.0};
  for (int i = threadIdx.x; i < P / 2; i += blockDim.x)
    s[0] += w.q[i] * (key_value(keys[i]) - key_value(keys[P - 1 - i]));
  block_sum<1>(s, scratch);
  if (threadIdx.x == 0) w.xq[f] = s[0];
}

// The same for systems above MP_R_MAX_PATHS paths, whose keys (2 P at most)
// lie in ReduceParams::sort_buf: tiles of MP_R_MAX_PATHS keys in shared
// memory, strides above a tile through memory, one launch per step and one
// field at a time.
//   k = 0: load the field and sort each tile;  stride >= tile: one global
//   step;  stride < tile: the remaining strides of stage k in each tile.
__device__ bool large_system(const ReduceParams& p, const DevSystem& sy) {
  return sy.n_paths > MP_R_MAX_PATHS && sy.n_paths <= (int64_t{1} << 30) && p.sort_buf != nullptr;
}
__global__ void __launch_bounds__(kSortThreads) sort_tiles_kernel(const ReduceParams p, int f, int64_t k) {
  extern __shared__ __align__(16) int64_t keys[];
  const DevSystem& sy = p.systems[blockIdx.y];
  if (!large_system(p, sy)) return;
  const int64_t P = sy.n_paths, n = pow2_above(P);
  if (k > n) return;
  int64_t* buf = reinterpret_cast<int64_t*>(p.sort_buf) + 2 * sy.rec_offset;
  const double* x = p.records + sy.rec_offset * MP_NREC + kRField[f];
  constexpr int kTile = MP_R_MAX_PATHS;
  for (int64_t tile = blockIdx.x; tile < n / kTile; tile += gridDim.x) {
    const int64_t base = tile * kTile;
    for (int i = threadIdx.x; i < kTile; i += blockDim.x)
      keys[i] = k ? buf[base + i] : order_key(base + i < P ? x[(base + i) * MP_NREC] : INFINITY);
    __syncthreads();
    if (k) bitonic_strides(keys, kTile, base, k, kTile / 2);
    else
      for (int q = 2; q <= kTile; q <<= 1) bitonic_strides(keys, kTile, base, q, q >> 1);
    for (int i = threadIdx.x; i < kTile; i += blockDim.x) buf[base + i] = keys[i];
    __syncthreads();
  }
}
__global__ void sort_step_kernel(const ReduceParams p, int64_t k, int64_t j) {
  const DevSystem& sy = p.systems[blockIdx.y];
  if (!large_system(p, sy)) return;
  const int64_t n = pow2_above(sy.n_paths);
  if (k > n) return;
  int64_t* buf = reinterpret_cast<int64_t*>(p.sort_buf) + 2 * sy.rec_offset;
  for (int64_t t = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; t < n / 2;
       t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t i = 2 * t - (t & (j - 1));
    const int64_t a = buf[i], b = buf[i + j];
    if ((a > b) == ((i & k) == 0)) {
      buf[i] = b;
      buf[i + j] = a;
    }
  }
}
__global__ void __launch_bounds__(kRedThreads) sort_fit_kernel(const ReduceParams p, int f) {
  __shared__ double scratch[kRedThreads / 32];
  const DevSystem& sy = p.systems[blockIdx.y];
  const int64_t P = sy.n_paths;
  const int nb = reduce_ctas(P);
  if (!large_system(p, sy) || static_cast<int>(blockIdx.x) >= nb) return;
  const ReduceScratch w(p, blockIdx.y, sy.rec_offset, P);
  const int64_t* buf = reinterpret_cast<const int64_t*>(p.sort_buf) + 2 * sy.rec_offset;
  double s[1] = {0.0};
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * kRedThreads + threadIdx.x; i < P / 2; i += nb * kRedThreads)
    s[0] += w.q[i] * (key_value(buf[i]) - key_value(buf[P - 1 - i]));
  block_sum<1>(s, scratch);
  if (threadIdx.x == 0) w.xq[blockIdx.x * kNumR + f] = s[0];
}

// Pass 2: variances, half variances and jackknife; the last CTA of a system
// to finish writes its estimates.
__global__ void __launch_bounds__(kRedThreads) reduce_finish_kernel(const ReduceParams p) {
  __shared__ TotalBuf<kVars> buf;
  __shared__ double tot[kSums], var[kVars], xq[kNumR];
  __shared__ bool last;
  const int sidx = blockIdx.y;
  const DevSystem& sy = p.systems[sidx];
  const int64_t P = sy.n_paths;
  const int nb = reduce_ctas(P), tid = threadIdx.x;
  if (static_cast<int>(blockIdx.x) >= nb) return;
  const ReduceScratch w(p, sidx, sy.rec_offset, P);
  const double* rec = p.records + sy.rec_offset * MP_NREC;
  const double N = static_cast<double>(sy.N), beta = sy.beta;
  const double invP = 1.0 / static_cast<double>(P);
  const int64_t Pa = P - P / 2, Pb = P / 2;
  if (tid < kSums) {
    double t = w.sums[tid];
    for (int c = 1; c < nb; ++c) {
      const double u = w.sums[c * kSums + tid];
      t = tid == kSums - 1 ? fmax(t, u) : t + u;
    }
    tot[tid] = t;
  }
  __syncthreads();
  double mu[kNumMean + 1];
#pragma unroll
  for (int k = 0; k <= kNumMean; ++k) mu[k] = tot[k] * invP;
  const double hmu[4] = {tot[kNumMean + 1] / Pa, tot[kNumMean + 2] / Pa, Pb ? tot[kNumMean + 3] / Pb : NAN,
                         Pb ? tot[kNumMean + 4] / Pb : NAN};
  double th_full[kNumDerived];
  derived(mu, N, beta, th_full);
  double v[kVars];
#pragma unroll
  for (int k = 0; k < kVars; ++k) v[k] = 0.0;
  double own[kNumDerived];  // delete-one values of this thread's last path
#pragma unroll
  for (int k = 0; k < kNumDerived; ++k) own[k] = 0.0;
  const bool jk = P >= 2;
  const double invPm1 = jk ? 1.0 / static_cast<double>(P - 1) : 0.0;
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * kRedThreads + tid; i < P; i += nb * kRedThreads) {
    const double* r = rec + i * MP_NREC;
    double loo[kNumMean], th[kNumDerived];
#pragma unroll
    for (int k = 0; k < kNumMean; ++k) {
      const double x = r[k], d = x - mu[k];
      v[k] += d * d;
      loo[k] = (tot[k] - x) * invPm1;
    }
    const double da = r[MP_R_ACC] - mu[kNumMean];
    v[kNumMean] += da * da;
    const bool a = i < Pa;
    const double de = r[MP_R_E] - (a ? hmu[0] : hmu[2]), dm = r[MP_R_M] - (a ? hmu[1] : hmu[3]);
    const double e2 = de * de, m2 = dm * dm;
    v[kNumMean + 1] += a ? e2 : 0.0;
    v[kNumMean + 2] += a ? m2 : 0.0;
    v[kNumMean + 3] += a ? 0.0 : e2;
    v[kNumMean + 4] += a ? 0.0 : m2;
    if (jk) {
      // delete-one values about the full estimate: their mean is O(1/P^2)
      // and their spread O(1/P) away from it, so for many paths sums and
      // squares in one pass lose nothing
      derived(loo, N, beta, th);
#pragma unroll
      for (int k = 0; k < kNumDerived; ++k) {
        const double d = th[k] - th_full[k];
        own[k] = d;
        v[kNumMean + 5 + k] += d;
        v[kNumMean + 5 + kNumDerived + k] += d * d;
      }
    }
  }
  block_total<kVars>(v, buf);
  if (nb == 1 && jk) {  // few paths, one to a thread: squares about the mean itself
#pragma unroll
    for (int k = 0; k < kNumDerived; ++k) {
      const double d = tid < P ? own[k] - buf.total[kNumMean + 5 + k] * invP : 0.0;
      v[kNumMean + 5 + k] = 0.0;
      v[kNumMean + 5 + kNumDerived + k] = d * d;
    }
    __syncthreads();
    block_total<kVars>(v, buf);
  }
  if (tid < kVars) {
    w.vars[blockIdx.x * kVars + tid] = buf.total[tid];
    __threadfence();
  }
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    last = atomicAdd(w.done, 1u) + 1u == static_cast<unsigned>(nb);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (tid < kVars) {
    double t = 0.0;
    for (int c = 0; c < nb; ++c) t += __ldcg(w.vars + c * kVars + tid);
    var[tid] = t;
  } else if (tid >= 64 && tid < 64 + kNumR) {
    const int f = tid - 64;
    double t = NAN;
    if (P >= 3 && P <= MP_R_MAX_PATHS) {
      t = w.xq[f];
    } else if (large_system(p, sy)) {
      t = 0.0;
      for (int c = 0; c < nb; ++c) t += w.xq[c * kNumR + f];
    }
    xq[f] = t;
  }
  __syncthreads();
  // one lane per estimate: each square root and division is issued once
  mp_estimates_t* o = reinterpret_cast<mp_estimates_t*>(p.est + static_cast<int64_t>(sidx) * MP_NEST);
  const double dP = static_cast<double>(P);
  if (tid < 11) {  // e, e2, m, m2, m4, mx, my, mz, mz2, |mz|, acceptance
    const int k = tid < 10 ? tid : kNumMean;
    (&o->e)[2 * tid] = tot[k] * invP;
    (&o->e)[2 * tid + 1] = P >= 2 ? sqrt(var[k]) / sqrt(dP * (dP - 1.0)) : NAN;
  } else if (tid >= 32 && tid < 32 + kNumDerived) {
    const int k = tid - 32;
    const double s1 = var[kNumMean + 5 + k], s2 = var[kNumMean + 5 + kNumDerived + k];
#pragma unroll
    for (int j = 0; j < kNumDerived; ++j)
      if (j == k) (&o->chi)[2 * k] = th_full[j];
    // (a maximum that keeps NaN)
    double ss = s2 - s1 * s1 * invP;
    if (ss < 0.0) ss = 0.0;
    (&o->chi)[2 * k + 1] = jk ? sqrt((dP - 1.0) * invP * ss) : NAN;
  } else if (tid >= 64 && tid < 64 + kNumR) {
    const double sxx = var[kRField[tid - 64]], sqq = tot[kSums - 2], sxq = xq[tid - 64];
    (&o->r_e)[tid - 64] = sxx > 0.0 && sqq > 0.0 ? sxq * sxq / (sxx * sqq) : NAN;
  } else if (tid >= 96 && tid < 100) {
    const int k = tid - 96;  // e and |m| of the first half, then of the second
    const double n = static_cast<double>(k < 2 ? Pa : Pb);
    double* out = (k & 1 ? &o->m_a : &o->e_a) + (k < 2 ? 0 : 2);
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (j == k) out[0] = hmu[j];
    out[1] = n >= 2.0 ? sqrt(var[kNumMean + 1 + k] / (n * (n - 1.0))) : NAN;
  }
  __syncthreads();
  if (tid == 0) {
    o->n_paths = dP;
    o->N = N;
    o->T = sy.T;
    o->n_meas = static_cast<double>(p.n_meas);
    o->attempts = N * dP * static_cast<double>(p.n_therm + p.n_meas);
    o->norm_max = tot[kSums - 1];
    o->elapsed_s = NAN;  // the host fills it in from the run's events
    o->reserved[0] = 0.0;
  } else if (tid == 32) {
    o->cv_m = o->m_se / o->m;
  } else if (tid == 64) {
    const double ze = fabs(o->e_a - o->e_b) / sqrt(o->e_a_se * o->e_a_se + o->e_b_se * o->e_b_se);
    const double zm = fabs(o->m_a - o->m_b) / sqrt(o->m_a_se * o->m_a_se + o->m_b_se * o->m_b_se);
    o->start_z = fmax(ze, zm);  // an undefined ratio (0/0) is skipped
  }
}

// Covariance backward: for each system, with upstream gradients (g_e, g_m) of
// (<e>, <|m|>),  dL/dbeta = -N [g_e cov(e, e) + g_m cov(|m|, e)]  and
// dL/dh = beta N [g_e cov(e, m_z) + g_m cov(|m|, m_z)] - g_e <m_z> (the last
// term from the field part of e), covariances of the pooled per-path moments
// (the C_V / chi estimators of Eq. (cv)).
__global__ void __launch_bounds__(kBackThreads) backward_kernel(const BackwardParams p) {
  __shared__ double scratch[32 * 8];
  const int sidx = blockIdx.x;
  const DevSystem sy = p.systems[sidx];
  const int64_t P = sy.n_paths;
  const double* rec = p.records + sy.rec_offset * MP_NREC;
  double s[7] = {0, 0, 0, 0, 0, 0, 0};
  for (int64_t i = threadIdx.x; i < P; i += blockDim.x) {
    const double* r = rec + i * MP_NREC;
    s[0] += r[MP_R_E];
    s[1] += r[MP_R_E2];
    s[2] += r[MP_R_M];
    s[3] += r[MP_R_EM];
    s[4] += r[MP_R_MZ];
    s[5] += r[MP_R_EMZ];
    s[6] += r[MP_R_MMZ];
  }
  block_sum<7>(s, scratch);
  if (threadIdx.x == 0) {
    const double inv = 1.0 / static_cast<double>(P);
    const double e = s[0] * inv, e2 = s[1] * inv, m = s[2] * inv, em = s[3] * inv;
    const double mz = s[4] * inv, emz = s[5] * inv, mmz = s[6] * inv;
    const double N = static_cast<double>(sy.N), beta = sy.beta;
    const double ge = p.g_e[sidx], gm = p.g_m[sidx];
    p.grad_beta[sidx] = -N * (ge * (e2 - e * e) + gm * (em - m * e));
    p.grad_h[sidx] = beta * N * (ge * (emz - e * mz) + gm * (mmz - m * mz)) - ge * mz;
  }
}

__global__ void philox_kernel(const uint32_t* ctr, int64_t n, const PhiloxKeys key, uint32_t* out) {
  for (int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const Philox4 r = philox4x32_10(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3], key);
    out[4 * i] = r.x;
    out[4 * i + 1] = r.y;
    out[4 * i + 2] = r.z;
    out[4 * i + 3] = r.w;
  }
}

// Doubles of ReduceParams::work for a batch.
int64_t reduce_work_doubles(int64_t total_paths, int n_systems) {
  return total_paths + 64 * static_cast<int64_t>(n_systems);
}

cudaError_t launch_reduce(const ReduceParams& p, int n_systems, int64_t max_paths, cudaStream_t st) {
  const dim3 grid(static_cast<unsigned>(reduce_ctas(max_paths)), static_cast<unsigned>(n_systems));
  reduce_sums_kernel<<<grid, kRedThreads, 0, st>>>(p);
  int64_t n = 1;
  while (n < max_paths) n <<= 1;
  const int tile = static_cast<int>(n < MP_R_MAX_PATHS ? n : MP_R_MAX_PATHS);
  const int smem = tile * static_cast<int>(sizeof(int64_t));
  reduce_sort_kernel<<<dim3(kNumR, n_systems), kSortThreads, smem, st>>>(p);
  if (n > MP_R_MAX_PATHS && p.sort_buf != nullptr) {
    const int64_t tiles = n / MP_R_MAX_PATHS;
    const dim3 tgrid(static_cast<unsigned>(tiles < 152 ? tiles : 152), static_cast<unsigned>(n_systems));
    for (int f = 0; f < kNumR; ++f) {
      sort_tiles_kernel<<<tgrid, kSortThreads, smem, st>>>(p, f, 0);
      for (int64_t k = 2 * MP_R_MAX_PATHS; k <= n && k <= (int64_t{1} << 30); k <<= 1) {
        for (int64_t j = k >> 1; j >= MP_R_MAX_PATHS; j >>= 1)
          sort_step_kernel<<<dim3(152, n_systems), 512, 0, st>>>(p, k, j);
        sort_tiles_kernel<<<tgrid, kSortThreads, smem, st>>>(p, f, k);
      }
      sort_fit_kernel<<<grid, kRedThreads, 0, st>>>(p, f);
    }
  }
  reduce_finish_kernel<<<grid, kRedThreads, 0, st>>>(p);
  return cudaGetLastError();
}

// Raises the sorts' dynamic shared memory limit.
cudaError_t reduce_prepare() {
  const int bytes = MP_R_MAX_PATHS * static_cast<int>(sizeof(int64_t));
  const cudaError_t e = cudaFuncSetAttribute(reduce_sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(sort_tiles_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

cudaError_t launch_backward(const BackwardParams& p, int n_systems, cudaStream_t st) {
  backward_kernel<<<n_systems, kBackThreads, 0, st>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_philox(const uint32_t* ctr, int64_t n, uint64_t seed, uint32_t* out,
                          cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  const int threads = 256;
  int64_t blocks = (n + threads - 1) / threads;
  if (blocks > 4096) blocks = 4096;
  philox_kernel<<<static_cast<int>(blocks), threads, 0, st>>>(ctr, n, philox_round_keys(seed), out);
  return cudaGetLastError();
}

}  // namespace mpk
