// The paper's literal sweep order (Sec. 2.2): a lattice sweep is N Metropolis
// attempts at randomly chosen sites, so consecutive attempts of one path may
// touch neighbouring sites and must act in order.
//
// Attempt a of sweep s of a path draws one counter (a, s, path, 2 | sys<<8):
// the site is the cell of width 1/N holding u(r3), i = floor((2 r3 + 1) N / 2^33)
// in integer arithmetic, and r0, r1, r2 drive the trial move and the accept
// test exactly as in the checkerboard kernels.  After every measurement sweep
// the energy is a bond loop (+x, +y, +z bonds of each site, in site order) and
// m the spin sum, in the working precision (FP64 form: exact integer sums).
//
// GB300 mapping: one warp per path, 32 consecutive attempts at a time.  Which
// sites they visit, their trial directions and their uniforms do not depend on
// the spins, so the lanes draw them together; only an attempt whose site is,
// or neighbours, the site of an earlier attempt of the 32 has to wait for it.
// Each lane marks its site in a table of lane masks and collects the earlier
// lanes among the marks of its site and neighbours; attempts then act in
// rounds, each round those with nobody left to wait for (the lowest waiting
// lane always is one, so at most 32 rounds; 2 to 3 at N = 1000).  Any order
// that respects these waits gives the sequential result, bit for bit.  What
// bounds it are shared-memory wavefronts of the seven scattered spin loads.
// L = 10, 10^4 paths, 10 + 10 sweeps: 82.4 ms with one thread per path and
// lattices in HBM, 4.6 ms so.
//
// The lattice is in shared memory where enough paths share an SM
// (shared_paths), otherwise in HBM (path by path, L2 holding what it can).
#include <algorithm>

#include "kernels.h"
#include "sweep.cuh"

namespace mpk {

namespace {

constexpr uint32_t kTagSite = 2u;
constexpr int kSlots = 512;        // lane masks; sites share a slot modulo kSlots (a false wait at worst)
constexpr int kDots = 208;         // floats of measure()'s products
constexpr int kWarps = 8;          // paths per CTA at most
// Paths that must fit an SM's shared memory for the lattices to live there.
// FP32: shared memory wins even at one path per SM (L = 26: 7.2e9 against
// 4.0e9 attempts/s; L = 10: 6.3e10 against 3.8e10).  FP64, with 24 bytes a
// spin: at 8 paths (L = 10: 2.5e10 against 2.0e10), not at 5 (L = 12: 1.6e10
// against 2.0e10).
constexpr int shared_paths(int real) { return real == 8 ? 6 : 1; }

// A path's spins by site: in shared memory as (x, y) pairs and z, in HBM as
// one float4 (FP32) or three consecutive integers (FP64) per site.
template <typename Real, bool kShared>
struct SiteStore {
  SpinView<Real> v;
  __device__ SiteStore(void* base, int N) : v(static_cast<Real*>(base), N) {}
  __device__ __forceinline__ V3<Real> ld(int i) const { return v.ld(i); }
  __device__ __forceinline__ void st(int i, V3<Real> s) const { v.st(i, s.x, s.y, s.z); }
};
template <>
struct SiteStore<float, false> {
  float4* a;
  __device__ SiteStore(void* base, int) : a(static_cast<float4*>(base)) {}
  __device__ __forceinline__ V3<float> ld(int i) const {
    const float4 v = a[i];
    return V3<float>{v.x, v.y, v.z};
  }
  __device__ __forceinline__ void st(int i, V3<float> s) const { a[i] = make_float4(s.x, s.y, s.z, 0.f); }
};
template <>
struct SiteStore<double, false> {
  int64_t* a;
  __device__ SiteStore(void* base, int) : a(static_cast<int64_t*>(base)) {}
  __device__ __forceinline__ V3<double> ld(int i) const {
    const int64_t* p = a + 3 * static_cast<int64_t>(i);
    return V3<double>{p[0], p[1], p[2]};
  }
  __device__ __forceinline__ void st(int i, V3<double> s) const {
    int64_t* p = a + 3 * static_cast<int64_t>(i);
    p[0] = s.x;
    p[1] = s.y;
    p[2] = s.z;
  }
};

// i / L for i < 2^31, M = floor(2^32 / L) + 1: the product overshoots by one at most.
__device__ __forceinline__ int div_by(int i, int L, uint32_t M) {
  const int q = static_cast<int>(__umulhi(static_cast<uint32_t>(i), M));
  return i - q * L < 0 ? q - 1 : q;
}

// Neighbours of site i in the fixed order +x, -x, +y, -y, +z, -z (simple
// cubic, periodic) or i-1, i+1 where they exist (open chain); returns how many.
template <bool kChain>
__device__ __forceinline__ int neighbours(int L, uint32_t M, int i, int* nb) {
  if constexpr (kChain) {
    const bool lo = i > 0, hi = i < L - 1;
    nb[0] = lo ? i - 1 : i + 1;
    nb[1] = i + 1;
    return static_cast<int>(lo) + static_cast<int>(hi);
  } else {
    const int t = div_by(i, L, M), x = i - t * L, z = div_by(t, L, M), y = t - z * L;
    const int LL = L * L;
    nb[0] = i + (x == L - 1 ? 1 - L : 1);
    nb[1] = i + (x == 0 ? L - 1 : -1);
    nb[2] = i + (y == L - 1 ? L - LL : L);
    nb[3] = i + (y == 0 ? LL - L : -L);
    nb[4] = i + (z == L - 1 ? -(L - 1) * LL : LL);
    nb[5] = i + (z == 0 ? (L - 1) * LL : -LL);
    return 6;
  }
}

// One attempt's draws, and its accept test once the local field f and the
// spin a are known: true with the new spin in n.
template <typename Real>
struct Attempt;
template <>
struct Attempt<float> {
  float tx, ty, tz;
  uint32_t r2;
  __device__ __forceinline__ explicit Attempt(const Philox4& r) : r2(r.z) { Arith<float>::trial(r.x, r.y, tx, ty, tz); }
  __device__ __forceinline__ bool test(V3<float> a, V3<float> f, const Couplings<float>& cp, V3<float>& n) const {
    n = V3<float>{tx, ty, tz};
    using A = Arith<float>;
    return A::accept_move(A::sub(tx, a.x), A::sub(ty, a.y), A::sub(tz, a.z), f.x, f.y, f.z, cp.J, cp.hf, cp.bp, r2);
  }
};
template <>
struct Attempt<double> {
  Philox4 r;
  __device__ __forceinline__ explicit Attempt(const Philox4& r_) : r(r_) {}
  __device__ __forceinline__ bool test(V3<double> a, V3<double> f, const Couplings<double>& cp, V3<double>& n) const {
    bool ok = false;
    move_fixed(r, a, f, cp, [&](V3<double> t) {
      n = t;
      ok = true;
    });
    return ok;
  }
};

// f / N correctly rounded, for f an FP32 number and invN = 1 / N correctly
// rounded: the product's residual is exact and corrects it (P. Markstein, IBM J.
// Res. Dev. 34, 1990); f / N keeps 2^-31 of an ulp from every midpoint of two
// doubles (f has 24 bits and N fewer than 31), far more than what is neglected.
// Three FP64 instructions of 76 cycles each instead of a division's ten.
__device__ __forceinline__ double per_site(double f, double dN, double invN) {
  const double q = __dmul_rn(f, invN);
  if ((__double2hiint(q) & 0x7ff00000) == 0x7ff00000) return q;  // infinity, NaN
  return __fma_rn(__fma_rn(-q, dN, f), invN, q);
}

// Sums of one measurement: bonds and spins over all sites.  FP32: added one
// by one in site order (lane 0 the bonds, lanes 1 to 3 a component each, from
// the dot products that the 32 lanes leave in `dots`), so that the sums are
// those of a plain loop over the sites.
template <bool kChain, class Store>
__device__ void measure(const Store& S, int N, int L, uint32_t M, int lane, float* dots, Partials<float>& part) {
  constexpr int D = kChain ? 1 : 3;
  // where the dot products (0) and the components (1, 2, 3) start: four
  // lanes read four arrays, 16 bytes each, on different banks
  auto at = [](int k) { return k == 0 ? 0 : 32 * D + 4 + 36 * (k - 1); };
  float sum = 0.f;
  for (int i0 = 0; i0 < N; i0 += 32) {
    const int i = i0 + lane, cnt = min(32, N - i0);
    V3<float> a{};
    if (i < N) {
      a = S.ld(i);
      int nb[6];
      neighbours<kChain>(L, M, i, nb);
#pragma unroll
      for (int d = 0; d < D; ++d) {
        if (!kChain || i + 1 < N) {
          const V3<float> b = S.ld(nb[kChain ? 1 : 2 * d]);
          dots[lane * D + d] = a.x * b.x + a.y * b.y + a.z * b.z;
        }
      }
      dots[at(1) + lane] = a.x;
      dots[at(2) + lane] = a.y;
      dots[at(3) + lane] = a.z;
    }
    __syncwarp();
    const float* src = dots + at(min(lane, 3));
    const int n = lane == 0 ? (kChain ? min(cnt, N - 1 - i0) : cnt * D) : cnt;
    if (lane < 4) {
      if (n % 32 == 0) {
        for (int k = 0; k < n; k += 32) {
          float4 v[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) v[j] = reinterpret_cast<const float4*>(src + k)[j];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            sum += v[j].x;
            sum += v[j].y;
            sum += v[j].z;
            sum += v[j].w;
          }
        }
      } else {
        for (int k = 0; k < n; ++k) sum += src[k];
      }
    }
    __syncwarp();
  }
  part.eb = __shfl_sync(0xffffffffu, sum, 0);
  part.mx = __shfl_sync(0xffffffffu, sum, 1);
  part.my = __shfl_sync(0xffffffffu, sum, 2);
  part.mz = __shfl_sync(0xffffffffu, sum, 3);
}
// FP64 form: exact integer sums, in any order.
template <bool kChain, class Store>
__device__ void measure(const Store& S, int N, int L, uint32_t M, int lane, float*, Partials<double>& part) {
  for (int i = lane; i < N; i += 32) {
    const V3<double> a = S.ld(i);
    part.mx.add(a.x);
    part.my.add(a.y);
    part.mz.add(a.z);
    int nb[6];
    neighbours<kChain>(L, M, i, nb);
#pragma unroll
    for (int d = 0; d < (kChain ? 1 : 3); ++d) {
      if (!kChain || i + 1 < N) {
        const V3<double> b = S.ld(nb[kChain ? 1 : 2 * d]);
        part.eb.add(spin_dot(a, b));
      }
    }
  }
}

template <typename Real, bool kShared, bool kChain>
__device__ void run_path_random(const DevSystem* sy, int sys_idx, int64_t path, int64_t gp, const SweepParams& P,
                                void* spins, uint32_t* marks, float* dots, int lane) {
  const int N = sy->N, L = sy->L;
  const uint32_t M = static_cast<uint32_t>((uint64_t{1} << 32) / static_cast<uint32_t>(L)) + 1u;
  const SiteStore<Real, kShared> S(spins, (N + 1) & ~1);
  const uint32_t c2 = static_cast<uint32_t>(sy->path_begin + path);  // path id
  const uint32_t sys_hi = static_cast<uint32_t>(sys_idx) << 8;
  const int init = path_init_mode(P.init_mode, path, sy->n_paths);
  for (int k = lane; k < kSlots; k += 32) marks[k] = 0u;
  for (int i = lane; i < N; i += 32)
    S.st(i, initial_spin<Real>(static_cast<uint32_t>(i), c2, kTagInit | sys_hi, P, init));
  __syncwarp();
  const Couplings<Real> cp(sy);
  double acc = 0.0;  // lane k: record field k
  int64_t accepted = 0;
  const uint32_t before = (1u << lane) - 1u;
  const double dN = static_cast<double>(N), invN = __drcp_rn(dN);
  const int64_t S_total = P.n_therm + P.n_meas;
  for (int64_t s = 0; s < S_total; ++s) {
    const PhiloxPrefix pre = philox_prefix(static_cast<uint32_t>(s), c2, kTagSite | sys_hi, P.key);
    for (int a0 = 0; a0 < N; a0 += 32) {
      const int a = a0 + lane;
      const bool active = a < N;
      const Philox4 r = philox4x32_10(static_cast<uint32_t>(a), pre, P.key);
      const int i = static_cast<int>(((static_cast<uint64_t>(r.w) * 2u + 1u) * static_cast<uint64_t>(N)) >> 33);
      int nb[6];
      const int nn = neighbours<kChain>(L, M, i, nb);
      const Attempt<Real> at(r);
      if (active) atomicOr(&marks[i & (kSlots - 1)], 1u << lane);
      __syncwarp();
      uint32_t wait = marks[i & (kSlots - 1)];
#pragma unroll
      for (int j = 0; j < (kChain ? 2 : 6); ++j)
        if (j < nn) wait |= marks[nb[j] & (kSlots - 1)];
      wait &= before;
      __syncwarp();
      if (active) marks[i & (kSlots - 1)] = 0u;
      uint32_t pending = __ballot_sync(0xffffffffu, active);
      while (pending) {
        const bool ready = ((pending >> lane) & 1u) && !(wait & pending);
        if (ready) {
          V3<Real> f{};
#pragma unroll
          for (int j = 0; j < (kChain ? 2 : 6); ++j)
            if (j < nn) f = add3(f, S.ld(nb[j]));
          V3<Real> n;
          if (at.test(S.ld(i), f, cp, n)) {
            S.st(i, n);
            ++accepted;
          }
        }
        pending &= ~__ballot_sync(0xffffffffu, ready);
        __syncwarp();  // this round's spins are visible to the next
      }
    }
    if (s < P.n_therm) continue;
    Partials<Real> part;
    measure<kChain>(S, N, L, M, lane, dots, part);
    // e, m_x, m_y, m_z per site: lanes 0 to 3 divide one each
    double v;
    if constexpr (sizeof(Real) == 8) {
      // lanes 0 .. 3: bonds, M_x, M_y, M_z
      v = warp_sums(part.eb, part.my, part.mx, part.mz, lane).real(lane == 0 ? kEnergyBits : kFixBits);
      const double Mz = __shfl_sync(0xffffffffu, v, 3);
      if (lane == 0) v = __dsub_rn(__dmul_rn(-sy->J, v), __dmul_rn(sy->h, Mz));
    } else {
      const float en = -cp.J * part.eb - cp.hf * part.mz;
      v = static_cast<double>(lane == 0 ? en : lane == 1 ? part.mx : lane == 2 ? part.my : part.mz);
    }
    v = sizeof(Real) == 8 ? __ddiv_rn(v, dN) : per_site(v, dN, invN);
    const double e = __shfl_sync(0xffffffffu, v, 0), mx = __shfl_sync(0xffffffffu, v, 1),
                 my = __shfl_sync(0xffffffffu, v, 2), mz = __shfl_sync(0xffffffffu, v, 3);
    const double m = sqrt(__dadd_rn(__dadd_rn(__dmul_rn(mx, mx), __dmul_rn(my, my)), __dmul_rn(mz, mz)));
    // field k of the record is a product of at most two of these (m^4: m m m m)
    const bool is_m = lane == MP_R_M || lane == MP_R_M2 || lane == MP_R_M4 || lane == MP_R_MMZ;
    const double p = (lane == MP_R_E || lane == MP_R_E2 || lane == MP_R_EM || lane == MP_R_EMZ || lane == MP_R_FE) ? e
                     : is_m                                                                                     ? m
                     : (lane == MP_R_MX || lane == MP_R_FMX)                                                    ? mx
                     : (lane == MP_R_MY || lane == MP_R_FMY)                                                    ? my
                                                                                                                : mz;
    const double q = lane == MP_R_E2                                                        ? e
                     : (lane == MP_R_M2 || lane == MP_R_M4 || lane == MP_R_EM)              ? m
                     : (lane == MP_R_MZ2 || lane == MP_R_EMZ || lane == MP_R_MMZ)           ? mz
                                                                                            : 1.0;
    double x = __dmul_rn(p, q);
    const double x4 = __dmul_rn(__dmul_rn(x, m), m);
    if (lane == MP_R_M4) x = x4;
    if (lane == MP_R_AMZ) x = fabs(mz);
    if (lane <= MP_R_MMZ) acc = __dadd_rn(acc, x);
    else if (s == S_total - 1) acc = x;
  }
  double worst = 0.0;
  double* out = P.spins ? P.spins + P.spin_offset[sys_idx] + path * 3 * static_cast<int64_t>(N) : nullptr;
  Real wst = Real(0);
  for (int i = lane; i < N; i += 32) {
    const V3<Real> v = S.ld(i);
    wst = fmax(wst, norm_error(v));
    if (out) {
      out[3 * i + 0] = Stored<Real>::real(v.x);
      out[3 * i + 1] = Stored<Real>::real(v.y);
      out[3 * i + 2] = Stored<Real>::real(v.z);
    }
  }
  worst = static_cast<double>(wst);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    accepted += __shfl_xor_sync(0xffffffffu, accepted, o);
    worst = fmax(worst, __shfl_xor_sync(0xffffffffu, worst, o));
  }
  double rv = acc;
  if (lane <= MP_R_MMZ) rv = __ddiv_rn(acc, static_cast<double>(P.n_meas));
  if (lane == MP_R_ACC) rv = static_cast<double>(accepted) / (static_cast<double>(S_total) * static_cast<double>(N));
  if (lane == MP_R_NORM) rv = worst;
  if (lane == MP_R_SPARE) rv = 0.0;
  if (lane < MP_NREC) P.records[gp * MP_NREC + lane] = rv;
  __syncwarp();  // the slice is reused by the warp's next path
}

// The system of global path gp: the last one whose first path is <= gp.
__device__ __forceinline__ int system_of_path(const DevSystem* systems, int n_systems, int64_t gp) {
  int lo = 0, hi = n_systems - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (systems[mid].rec_offset <= gp) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Bytes of one warp's slice: lane masks, dot products, spins.
__host__ __device__ constexpr int slice_head() { return kSlots * 4 + kDots * 4; }
constexpr int64_t slice_bytes(int real, int64_t N, bool shared) {
  return (slice_head() + (shared ? 3 * ((N + 1) & ~int64_t{1}) * real : 0) + 15) / 16 * 16;
}

template <typename Real, bool kShared>
__global__ void __launch_bounds__(32 * kWarps) random_site_kernel(const SweepParams P, int n_systems,
                                                                  int64_t total_paths, void* lattice, int slice) {
  extern __shared__ __align__(16) unsigned char smem[];
  if constexpr (sizeof(Real) == 8) {
    for (int k = static_cast<int>(threadIdx.x); k < 256; k += static_cast<int>(blockDim.x))
      sine_shared()[k] = kSineTable.s[k];
    __syncthreads();
  }
  const int lane = threadIdx.x & 31;
  unsigned char* mine = smem + (threadIdx.x >> 5) * slice;
  uint32_t* marks = reinterpret_cast<uint32_t*>(mine);
  float* dots = reinterpret_cast<float*>(mine + kSlots * 4);
  for (;;) {
    unsigned long long next = 0;  // both words of the queue: paths, not work items
    if (lane == 0) next = atomicAdd(reinterpret_cast<unsigned long long*>(P.queue), 1ull);
    const int64_t gp = static_cast<int64_t>(__shfl_sync(0xffffffffu, next, 0));
    if (gp >= total_paths) return;
    const int lo = system_of_path(P.systems, n_systems, gp);
    const DevSystem* sy = P.systems + lo;
    const int64_t path = gp - sy->rec_offset;
    void* spins = mine + slice_head();
    if constexpr (!kShared)
      spins = static_cast<unsigned char*>(lattice) +
              (P.spin_offset[lo] / 3 + path * sy->N) * (sizeof(Real) == 4 ? 16 : 24);
    if (sy->lattice == MP_LATTICE_CHAIN)
      run_path_random<Real, kShared, true>(sy, lo, path, gp, P, spins, marks, dots, lane);
    else
      run_path_random<Real, kShared, false>(sy, lo, path, gp, P, spins, marks, dots, lane);
  }
}

// One thread per path, for many paths of very few sites (N <= kThreadSites),
// where 32 attempts of one path hardly ever act together: chain of 8, 10^4
// paths, FP32: 4.5e10 attempts/s against 2.3e10 by warps, measured sweeps
// 2.1e10 against 0.5e10; with 10^6 paths 1.8e11 against 2.5e10.  Lattices in HBM,
// element (site i, path p) of system k at spin_offset[k] / 3 + i * P_k + p, so
// that a warp's threads read consecutive elements of the same site.
constexpr int kThreadSites = 16;  // and enough paths for a warp of them on every SM

template <typename Real>
struct ColumnStore;
template <>
struct ColumnStore<float> {
  float4* a;
  int64_t stride;
  __device__ ColumnStore(void* lattice, int64_t base, int64_t stride_, int64_t)
      : a(static_cast<float4*>(lattice) + base), stride(stride_) {}
  __device__ __forceinline__ V3<float> ld(int i) const {
    const float4 v = a[i * stride];
    return V3<float>{v.x, v.y, v.z};
  }
  __device__ __forceinline__ void st(int i, V3<float> s) const { a[i * stride] = make_float4(s.x, s.y, s.z, 0.f); }
};
template <>
struct ColumnStore<double> {
  int64_t* a;
  int64_t stride, plane;  // three planes of components
  __device__ ColumnStore(void* lattice, int64_t base, int64_t stride_, int64_t plane_)
      : a(static_cast<int64_t*>(lattice) + base), stride(stride_), plane(plane_) {}
  __device__ __forceinline__ V3<double> ld(int i) const {
    const int64_t* p = a + i * stride;
    return V3<double>{p[0], p[plane], p[2 * plane]};
  }
  __device__ __forceinline__ void st(int i, V3<double> s) const {
    int64_t* p = a + i * stride;
    p[0] = s.x;
    p[plane] = s.y;
    p[2 * plane] = s.z;
  }
};

template <typename Real, bool kChain>
__device__ void run_path_thread(const DevSystem* sy, int sys_idx, int64_t path, int64_t gp, const SweepParams& P,
                                void* lattice, int64_t elements) {
  const int N = sy->N, L = sy->L;
  const uint32_t M = static_cast<uint32_t>((uint64_t{1} << 32) / static_cast<uint32_t>(L)) + 1u;
  const ColumnStore<Real> S(lattice, P.spin_offset[sys_idx] / 3 + path, sy->n_paths, elements);
  const uint32_t c2 = static_cast<uint32_t>(sy->path_begin + path);
  const uint32_t sys_hi = static_cast<uint32_t>(sys_idx) << 8;
  const int init = path_init_mode(P.init_mode, path, sy->n_paths);
  for (int i = 0; i < N; ++i) S.st(i, initial_spin<Real>(static_cast<uint32_t>(i), c2, kTagInit | sys_hi, P, init));
  const Couplings<Real> cp(sy);
  const double dN = static_cast<double>(N), invN = __drcp_rn(dN);
  double acc[MP_R_ACC];
#pragma unroll
  for (int q = 0; q < MP_R_ACC; ++q) acc[q] = 0.0;
  int64_t accepted = 0;
  const int64_t S_total = P.n_therm + P.n_meas;
  for (int64_t s = 0; s < S_total; ++s) {
    const PhiloxPrefix pre = philox_prefix(static_cast<uint32_t>(s), c2, kTagSite | sys_hi, P.key);
    for (int a = 0; a < N; ++a) {
      const Philox4 r = philox4x32_10(static_cast<uint32_t>(a), pre, P.key);
      const int i = static_cast<int>(((static_cast<uint64_t>(r.w) * 2u + 1u) * static_cast<uint64_t>(N)) >> 33);
      int nb[6];
      const int nn = neighbours<kChain>(L, M, i, nb);
      V3<Real> f{};
#pragma unroll
      for (int j = 0; j < (kChain ? 2 : 6); ++j)
        if (j < nn) f = add3(f, S.ld(nb[j]));
      V3<Real> n;
      if (Attempt<Real>(r).test(S.ld(i), f, cp, n)) {
        S.st(i, n);
        ++accepted;
      }
    }
    if (s < P.n_therm) continue;
    Partials<Real> part;  // bond loop and spin sum, in site order
    for (int i = 0; i < N; ++i) {
      const V3<Real> a = S.ld(i);
      int nb[6];
      neighbours<kChain>(L, M, i, nb);
      if constexpr (sizeof(Real) == 8) {
        part.mx.add(a.x);
        part.my.add(a.y);
        part.mz.add(a.z);
      } else {
        part.mx += a.x;
        part.my += a.y;
        part.mz += a.z;
      }
#pragma unroll
      for (int d = 0; d < (kChain ? 1 : 3); ++d) {
        if (!kChain || i + 1 < N) {
          const V3<Real> b = S.ld(nb[kChain ? 1 : 2 * d]);
          if constexpr (sizeof(Real) == 8) part.eb.add(spin_dot(a, b));
          else part.eb += a.x * b.x + a.y * b.y + a.z * b.z;
        }
      }
    }
    double e, mx, my, mz;
    if constexpr (sizeof(Real) == 8) {
      mz = part.mz.real() * kSpinUnit;
      e = __ddiv_rn(__dsub_rn(__dmul_rn(-sy->J, part.eb.real() * kEnergyUnit), __dmul_rn(sy->h, mz)), dN);
      mx = __ddiv_rn(part.mx.real() * kSpinUnit, dN);
      my = __ddiv_rn(part.my.real() * kSpinUnit, dN);
      mz = __ddiv_rn(mz, dN);
    } else {
      e = per_site(static_cast<double>(-cp.J * part.eb - cp.hf * part.mz), dN, invN);
      mx = per_site(static_cast<double>(part.mx), dN, invN);
      my = per_site(static_cast<double>(part.my), dN, invN);
      mz = per_site(static_cast<double>(part.mz), dN, invN);
    }
    const double m = sqrt(__dadd_rn(__dadd_rn(__dmul_rn(mx, mx), __dmul_rn(my, my)), __dmul_rn(mz, mz)));
    const double now[MP_R_ACC] = {e, __dmul_rn(e, e), m, __dmul_rn(m, m), __dmul_rn(__dmul_rn(__dmul_rn(m, m), m), m),
                                  mx, my, mz, __dmul_rn(mz, mz), fabs(mz), __dmul_rn(e, m), __dmul_rn(e, mz),
                                  __dmul_rn(m, mz), mx, my, mz, e};
#pragma unroll
    for (int q = 0; q < MP_R_ACC; ++q) acc[q] = q <= MP_R_MMZ ? __dadd_rn(acc[q], now[q]) : now[q];
  }
  double* rec = P.records + gp * MP_NREC;
#pragma unroll
  for (int q = 0; q < MP_R_ACC; ++q) rec[q] = q <= MP_R_MMZ ? __ddiv_rn(acc[q], static_cast<double>(P.n_meas)) : acc[q];
  rec[MP_R_ACC] = static_cast<double>(accepted) / (static_cast<double>(S_total) * dN);
  Real worst = Real(0);
  double* out = P.spins ? P.spins + P.spin_offset[sys_idx] + path * 3 * static_cast<int64_t>(N) : nullptr;
  for (int i = 0; i < N; ++i) {
    const V3<Real> v = S.ld(i);
    worst = fmax(worst, norm_error(v));
    if (out) {
      out[3 * i + 0] = Stored<Real>::real(v.x);
      out[3 * i + 1] = Stored<Real>::real(v.y);
      out[3 * i + 2] = Stored<Real>::real(v.z);
    }
  }
  rec[MP_R_NORM] = static_cast<double>(worst);
  rec[MP_R_SPARE] = 0.0;
}

static_assert(MP_R_FE + 1 == MP_R_ACC && MP_R_MMZ + 1 == MP_R_FMX, "sums, then the final state");

template <typename Real>
__global__ void __launch_bounds__(128) random_thread_kernel(const SweepParams P, int n_systems, int64_t total_paths,
                                                            void* lattice, int64_t elements) {
  if constexpr (sizeof(Real) == 8) {
    for (int k = static_cast<int>(threadIdx.x); k < 256; k += static_cast<int>(blockDim.x))
      sine_shared()[k] = kSineTable.s[k];
    __syncthreads();
  }
  const int64_t gp = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (gp >= total_paths) return;
  const int k = system_of_path(P.systems, n_systems, gp);
  const DevSystem* sy = P.systems + k;
  if (sy->lattice == MP_LATTICE_CHAIN)
    run_path_thread<Real, true>(sy, k, gp - sy->rec_offset, gp, P, lattice, elements);
  else
    run_path_thread<Real, false>(sy, k, gp - sy->rec_offset, gp, P, lattice, elements);
}

const void* kernel_of(int precision, bool shared) {
  if (precision == MP_FP64)
    return shared ? reinterpret_cast<const void*>(random_site_kernel<double, true>)
                  : reinterpret_cast<const void*>(random_site_kernel<double, false>);
  return shared ? reinterpret_cast<const void*>(random_site_kernel<float, true>)
                : reinterpret_cast<const void*>(random_site_kernel<float, false>);
}

}  // namespace

// Lattice bytes per site and path in HBM.
int random_site_bytes_per_site(int precision) { return precision == MP_FP64 ? 24 : 16; }

cudaError_t random_site_plan(int precision, int64_t max_sites, int64_t total_paths, int device, RandomSitePlan* plan) {
  int optin = 0, sms = 0;
  cudaError_t e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
  if (e != cudaSuccess) return e;
  plan->thread_per_path = max_sites <= kThreadSites && total_paths >= int64_t{32} * sms;
  if (plan->thread_per_path) {
    plan->shared = false;
    plan->slice = plan->smem = 0;
    plan->cta = 128;
    plan->grid = static_cast<int>((total_paths + 127) / 128);
    return cudaSuccess;
  }
  const int real = precision == MP_FP64 ? 8 : 4;
  const int room = optin - 4096;  // the kernel's static data and the CTAs' reserved kilobyte each
  plan->shared = slice_bytes(real, max_sites, true) * shared_paths(real) <= room;
  plan->slice = static_cast<int>(slice_bytes(real, max_sites, plan->shared));
  const void* k = kernel_of(precision, plan->shared);
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, room);
  // the paths per CTA that put the most on an SM (the fewest among equals)
  int per_sm = 0, most = 0;
  for (int w = 1; w <= kWarps && w <= total_paths && w * plan->slice <= room && e == cudaSuccess; ++w) {
    int blocks = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k, 32 * w, static_cast<size_t>(w) * plan->slice);
    if (blocks * w > most) {
      most = blocks * w;
      per_sm = blocks;
      plan->cta = 32 * w;
    }
  }
  if (e != cudaSuccess) return e;
  plan->smem = plan->cta / 32 * plan->slice;
  const int64_t ctas = (total_paths + plan->cta / 32 - 1) / (plan->cta / 32);
  plan->grid = static_cast<int>(std::min<int64_t>(ctas, static_cast<int64_t>(sms) * std::max(per_sm, 1)));
  return cudaSuccess;
}

// elements = sites x paths over all systems (the size of a component plane of
// the thread-per-path FP64 form)
cudaError_t launch_random_site(int precision, const RandomSitePlan& plan, const SweepParams& p, int n_systems,
                               int64_t total_paths, void* lattice, int64_t elements, cudaStream_t st) {
  if (plan.thread_per_path) {
    void* args[] = {const_cast<SweepParams*>(&p), &n_systems, &total_paths, &lattice, &elements};
    const void* k = precision == MP_FP64 ? reinterpret_cast<const void*>(random_thread_kernel<double>)
                                         : reinterpret_cast<const void*>(random_thread_kernel<float>);
    return cudaLaunchKernel(k, dim3(plan.grid), dim3(plan.cta), args, 0, st);
  }
  int slice = plan.slice;
  void* args[] = {const_cast<SweepParams*>(&p), &n_systems, &total_paths, &lattice, &slice};
  return cudaLaunchKernel(kernel_of(precision, plan.shared), dim3(plan.grid), dim3(plan.cta), args,
                          static_cast<size_t>(plan.smem), st);
}

}  // namespace mpk
