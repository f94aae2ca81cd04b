// Multipath Metropolis for the square-lattice Ising model (Appendix A of
// Rakic et al.: the same scheme -- many independent paths from random
// starts, each thermalised and measured -- applied to a model with a discrete
// symmetry, checked against the Onsager-Yang solution).
//
// H = -J sum_bonds s_i s_j - h sum_i s_i, s_i = +-1, on a periodic L x L
// lattice (L even), site i = x + L y, colour (x + y) mod 2.  A sweep tests a
// flip of every colour-0 site, then of every colour-1 site:
// dE = 2 s_i (J sum_nb s_j + h), accepted when dE <= 0, else iff
// u < exp(-beta dE) with u = (r + 1/2) 2^-32 for a Philox word r.
//
// GB300 mapping: a spin is a byte (1 up, 0 down), and the four rows 4j .. 4j+3
// of one colour at one x/2 = hx are one 32-bit word, a strip: word
// hx + (L/2) j of its colour.  One Philox call serves a strip: row y takes word
// y mod 4 of Philox(hx + (L/2) j, sweep, path, (4 + colour) | sys << 8).  The
// neighbours of a strip's four sites are bytes of five words of the other
// colour, put in place by three byte permutations and counted for all four
// sites by three additions.  Row 4j + k has x = 2 hx + ((k + colour) & 1), so
// the other colour's strip at the same place holds one x neighbour of each
// row, the other is in the strip at hx + 1 (odd x) or hx - 1 (even x), and the
// y neighbours are the same strip shifted by a row, completed from the strips
// at j + 1 and j - 1.
// Every dE > 0 that can occur (5 neighbour counts x 2 spins) has its acceptance
// turned, on the host and in FP64, into an integer threshold t with
// u < exp(-beta dE)  <=>  r < t,  so the device test is an integer compare and
// the trajectories equal the FP64 definition exactly.  The per-sweep energy
// (from the colour-1 counts, every bond once) and magnetisation are exact
// integers; they enter the FP64 per-path accumulators of the Heisenberg
// kernels' measurement ring, in the same record layout (m_x = m_y = 0, m_z = m).
// What bounds it is instruction issue, Philox half of it, and some spilled
// registers (64 per thread, for CTAs of up to 1024; 100 bytes of spill stores, 192
// of loads).  L = 60, four T x 10^4 paths: with a byte load per neighbour and 256
// threads per path 38.6 ms for 50 + 100 sweeps (5.6e11 attempts/s), 21.8 ms (9.9e11)
// with words and one warp per path.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "kernels.h"
#include "sweep.cuh"

namespace mpk {

namespace {

constexpr int kIsingThreads = 1024;
constexpr uint32_t kOnes = 0x01010101u;
// A thread counts its accepted flips in 32 bits; every kAcceptFold sweeps the
// warp's sum, still below 2^32, goes to the path's total in FP64 (exact to 2^53).
// (In a loop of its own: a 64-bit count per thread, or a test in the sweep loop,
// costs registers that the kernel does not have, L = 60 0.5%, L = 6 1.2%.)
constexpr uint32_t kAcceptFold = 1u << 15;
static_assert(uint64_t{kAcceptFold} * MP_ISING_MAX_L * MP_ISING_MAX_L < uint64_t{1} << 32, "all flips of a lattice");

// Blocks per segment for tp threads: the walk takes rounds x (q + what a
// segment's start costs, about 0.4 of a strip).
__host__ __device__ inline int ising_segment(int L, int tp) {
  const int HL = L / 2, JB = (L + 3) / 4;
  int best_q = 1, best = 0x7fffffff;
  for (int q = 1; q <= JB; ++q) {
    const int units = HL * ((JB + q - 1) / q);
    const int cost = (units + tp - 1) / tp * (5 * q + 2);
    if (cost <= best) {
      best = cost;
      best_q = q;
    }
  }
  return best_q;
}

// How a colour's strips are dealt out: each column of JB row blocks is cut into
// segments of q blocks, and the units (column, segment), numbered
// u = column + HL segment, go to the threads round by round.  Along a segment the
// x neighbours' offsets are fixed and two of the five words are already in
// registers.
struct StripWalk {
  int HL, JB, S;     // words per row block, row blocks, strips per colour
  int CW;            // words per colour: the strips and a copy of block 0 behind the last
  int q, units;      // blocks per segment, units
  int dh, dg;        // tp = dg HL + dh
  bool ragged;       // L % 4 == 2: the last row block has two rows
  __device__ StripWalk(int L, int tp, int q_)
      : HL(L >> 1), JB((L + 3) >> 2), S(HL * JB), CW(S + HL), q(q_), units(HL * ((JB + q_ - 1) / q_)),
        ragged((L & 3) != 0) {
    dg = tp / HL;
    dh = tp - dg * HL;
  }
};

struct IsingSums {
  uint32_t accepted;
  int up_own, up_nb, up_pairs;
};

// Flip tests of colour kC for this thread's strips.  table: shared-memory
// address of the 16 thresholds (entry 8 b + n for spin b and n neighbours up),
// a multiple of 128.  kWide: a threshold of 0 or 2^32 may both occur, so the
// test takes 64 bits; otherwise t > 0 and r <= t - 1 is tested in 32.
template <int kC, bool kWide, bool kMeas, bool kEnergy>
__device__ __forceinline__ void ising_half_sweep(const StripWalk& w, const PhiloxPrefix& pre, const PhiloxKeys& key,
                                                 uint32_t* __restrict__ own, const uint32_t* __restrict__ oth,
                                                 uint32_t table, int tid, int tp, int hx, int g, IsingSums& sum) {
  for (int u = tid; u < w.units; u += tp) {
    int t = hx + w.HL * (g * w.q);
    int end = min((g + 1) * w.q, w.JB);
    const bool short_end = w.ragged && end == w.JB;
    int left = end - g * w.q - (short_end ? 1 : 0);  // whole blocks
    const int dl = hx == 0 ? w.HL - 1 : -1, dr = hx == w.HL - 1 ? 1 - w.HL : 1;
    uint32_t o = oth[t];
    uint32_t lo = g == 0 ? oth[t + w.S - w.HL] : oth[t - w.HL];
    if (w.ragged && g == 0) lo <<= 16;  // row L - 1 is byte 1 of the last block
    const uint32_t *pt = oth + t + w.HL, *pl = oth + t + dl, *pr = oth + t + dr;
    uint32_t* po = own + t;
    uint32_t flips = 0, ups = 0;        // per byte, at most 64 strips of at most one each
    // one strip; kShort: the two rows of a ragged last block, whose upper
    // neighbour is row 0
    auto strip = [&](auto short_c) {
      constexpr bool kShort = decltype(short_c)::value;
      const Philox4 r = philox4x32_10(static_cast<uint32_t>(t), pre, key);
      const uint32_t hi = *pt;
      // the second x neighbour: rows of odd x from the right, of even x from the left
      const uint32_t xo = __byte_perm(*pl, *pr, kC ? 0x3614 : 0x7250);
      const uint32_t up = __byte_perm(o, hi, kShort ? 0x4441 : 0x4321);
      const uint32_t dn = __byte_perm(o, lo, 0x2107);
      uint32_t n = o + xo + up + dn;
      const uint32_t b = *po;
      // the table address of each site: low byte from ix, the rest from `table`
      const uint32_t ix = n * 8u + (b * 64u + (table & 0xffu) * kOnes);
      const uint32_t word[4] = {r.x, r.y, r.z, r.w};
      uint32_t flip = 0;
#pragma unroll
      for (int k = 0; k < (kShort ? 2 : 4); ++k) {
        const uint32_t at = __byte_perm(ix, table, 0x7650 + k);
        if constexpr (kWide) {
          uint64_t th;
          asm("ld.shared.u64 %0, [%1];" : "=l"(th) : "r"(at));
          if (static_cast<uint64_t>(word[k]) < th) flip += 1u << (8 * k);
        } else {
          uint32_t th;
          asm("ld.shared.u32 %0, [%1];" : "=r"(th) : "r"(at));
          if (word[k] <= th) flip += 1u << (8 * k);
        }
      }
      const uint32_t s = b ^ flip;
      *po = s;
      flips += flip;
      if (kMeas) ups += s;
      if (kEnergy) {
        if (kShort) n &= 0xffffu;
        sum.up_nb = __dp4a(n, kOnes, static_cast<uint32_t>(sum.up_nb));
        sum.up_pairs = __dp4a(n, s, static_cast<uint32_t>(sum.up_pairs));
      }
      lo = o;
      o = hi;
      t += w.HL;
      pt += w.HL;
      pl += w.HL;
      pr += w.HL;
      po += w.HL;
    };
    for (; left > 0; --left) strip(std::false_type{});
    if (short_end) strip(std::true_type{});
    if (g == 0) own[hx + w.S] = own[hx];  // read as row L's block in the next half-sweep
    sum.accepted = __dp4a(flips, kOnes, sum.accepted);
    if (kMeas) sum.up_own = __dp4a(ups, kOnes, static_cast<uint32_t>(sum.up_own));
    g += w.dg;
    hx += w.dh;
    if (hx >= w.HL) {
      hx -= w.HL;
      ++g;
    }
  }
}

__device__ void run_path_ising(const DevSystem& sy, int sys_idx, int64_t path,
                               const SweepParams& P, unsigned char* slice, int tid, int tp,
                               int bar) {
  const int L = sy.L, N = sy.N, NH = sy.NH;
  const StripWalk walk(L, tp, ising_segment(L, tp));
  const int HL = walk.HL;
  unsigned char* base = slice + slice_spin_offset(tp, sy.ring, kRedBytes);
  unsigned char* table_at = base + ((128u - (smem_addr(base) & 127u)) & 127u);
  uint32_t* sp = reinterpret_cast<uint32_t*>(base + kIsingThrBytes);  // strips of colour 0, then of colour 1
  const uint32_t c2 = static_cast<uint32_t>(sy.path_begin + path);  // path id
  const uint32_t sys_hi = static_cast<uint32_t>(sys_idx) << 8;
  const int init = path_init_mode(P.init_mode, path, sy.n_paths);
  const int64_t j_first = P.s_begin > P.n_therm ? P.s_begin - P.n_therm : 0;
  Meter<double> meter{reinterpret_cast<double*>(slice + slice_acc_offset()),
                      reinterpret_cast<double*>(slice + slice_red_offset()),
                      sy.ring, tp >> 5, tid & 31, tid >> 5, tid,
                      1.0 / static_cast<double>(N), sy.J, sy.h, j_first};
  meter.start();
  unsigned char* st = path_state(P, sys_idx, path);
  int8_t* st_spins = st ? reinterpret_cast<int8_t*>(st + kStateHeader) : nullptr;
  __shared__ int cancel_flag[kMaxGroups];
  const int gidx = bar - 1;

  // thresholds: entry 8 b + n; t - 1 in 32 bits when none is zero
  const unsigned long long* thr = P.ising_thr + sys_idx * 10;
  bool wide = false;
  for (int k = 0; k < 10; ++k) wide = wide || thr[k] == 0;
  if (tid < 10) {
    const int n = tid % 5, up = tid < 5 ? 1 : 0;
    reinterpret_cast<unsigned long long*>(table_at)[8 * up + n] = wide ? thr[tid] : thr[tid] - 1;
  }
  // initial or saved spins (saved as +-1 bytes [colour][half index x/2 + (L/2) y])
  const bool resume = P.resume && st;
  for (int t = tid; t < 2 * walk.CW; t += tp) {
    const int c = t >= walk.CW, u = t - c * walk.CW, jc = u / HL, hx = u - jc * HL;
    const int j = jc == walk.JB ? 0 : jc;
    uint32_t word = 0;
    for (int k = 0; k < 4 && 4 * j + k < L; ++k) {
      const int y = 4 * j + k, x = 2 * hx + ((k + c) & 1), i = x + L * y;
      bool up = true;
      if (resume) {
        up = st_spins[c * NH + (i >> 1)] > 0;
      } else if (init != MP_INIT_ORDERED) {
        // random start: the top bit of word 0 of the site's init counter
        up = !(philox4x32_10(static_cast<uint32_t>(i), 0u, c2, kTagInit | sys_hi, P.key).x >> 31);
      }
      word |= static_cast<uint32_t>(up) << (8 * k);
    }
    sp[t] = word;
  }
  if (tid < kAccDoubles) meter.acc[tid] = resume ? reinterpret_cast<const double*>(st)[tid] : 0.0;
  double accepted_before = resume ? reinterpret_cast<const double*>(st)[kAccDoubles] : 0.0;
  double* const accepted = meter.acc + MP_R_ACC;  // accepted flips of this call; the meter leaves the place alone
  if (tid == 0) cancel_flag[gidx] = 0;
  group_sync(tp, bar);

  // sites of one colour in this warp's strips
  int mine = 0;
  for (int u = tid; u < walk.units; u += tp) {
    const int j0 = u / HL * walk.q, j1 = min(j0 + walk.q, walk.JB);
    mine += 4 * (j1 - j0) - (walk.ragged && j1 == walk.JB ? 2 : 0);
  }
  const int warp_sites = __reduce_add_sync(0xffffffffu, mine);
  IsingSums sum{0, 0, 0, 0};
  bool canceled = false;
  const uint32_t c3a = (kTagIsing + 0u) | sys_hi, c3b = (kTagIsing + 1u) | sys_hi;
  uint32_t* sp0 = sp;
  uint32_t* sp1 = sp + walk.CW;
  const uint32_t table = smem_addr(table_at);
  const int g0 = tid / HL, h0 = tid - g0 * HL;
  auto sweep = [&](auto wide_c) {
    constexpr bool kWide = decltype(wide_c)::value;
    for (int64_t s = P.s_begin; s < P.s_end && !canceled;) {
      const uint32_t last = static_cast<uint32_t>(min(s | static_cast<int64_t>(kAcceptFold - 1), P.s_end - 1));
      for (;; ++s) {
        const uint32_t sw = static_cast<uint32_t>(s);
        const PhiloxPrefix pa = philox_prefix(sw, c2, c3a, P.key), pb = philox_prefix(sw, c2, c3b, P.key);
        sum.up_own = sum.up_nb = sum.up_pairs = 0;
        poll_cancel(P, s, tid, &cancel_flag[gidx]);
        const bool meas = s >= P.n_therm;
        if (meas)
          ising_half_sweep<0, kWide, true, false>(walk, pa, P.key, sp0, sp1, table, tid, tp, h0, g0, sum);
        else
          ising_half_sweep<0, kWide, false, false>(walk, pa, P.key, sp0, sp1, table, tid, tp, h0, g0, sum);
        group_sync(tp, bar);
        if (cancel_flag[gidx]) {
          canceled = true;
          break;
        }
        if (!meas) {
          ising_half_sweep<1, kWide, false, false>(walk, pb, P.key, sp1, sp0, table, tid, tp, h0, g0, sum);
          group_sync(tp, bar);
          if (sw == last) break;
          continue;
        }
        const int64_t j = s - P.n_therm;
        meter.maybe_flush(j);
        const int ups0 = sum.up_own;
        ising_half_sweep<1, kWide, true, true>(walk, pb, P.key, sp1, sp0, table, tid, tp, h0, g0, sum);
        // exact integers, then one slot of the ring: over the warp's sites
        // sum s = 2 (spins up) - sites, and over its colour-1 sites, with s = 2 b - 1
        // and neighbour sum 2 n - 4, sum s (2 n - 4) = 4 sum b n - 8 sum b - 2 sum n + 4 sites
        const int b1 = __reduce_add_sync(0xffffffffu, sum.up_own - ups0), b0 = __reduce_add_sync(0xffffffffu, ups0);
        const int nn = __reduce_add_sync(0xffffffffu, sum.up_nb), bn = __reduce_add_sync(0xffffffffu, sum.up_pairs);
        if ((tid & 31) == 0) {
          double* r = meter.cur_slot() + (tid >> 5) * kRedSlots;
          r[0] = static_cast<double>(4 * bn - 8 * b1 - 2 * nn + 4 * warp_sites);
          r[1] = 0.0;
          r[2] = 0.0;
          r[3] = static_cast<double>(2 * (b0 + b1) - 2 * warp_sites);
        }
        meter.advance();
        group_sync(tp, bar);
        if (sw == last) break;
      }
      ++s;
      const uint32_t flips = __reduce_add_sync(0xffffffffu, sum.accepted);
      if ((tid & 31) == 0) atomicAdd(accepted, static_cast<double>(flips));
      sum.accepted = 0;
    }
  };
  if (wide) sweep(std::true_type{});
  else sweep(std::false_type{});
  if (canceled) {
    group_sync(tp, bar);
    return;
  }
  auto spin_at = [&](int x, int y) {  // +-1
    const uint32_t word = sp[((x + y) & 1) * walk.CW + (y >> 2) * HL + (x >> 1)];
    return ((word >> (8 * (y & 3))) & 1u) ? 1 : -1;
  };
  const int64_t n_meas_done = P.s_end > P.n_therm ? P.s_end - P.n_therm : 0;
  meter.finish(n_meas_done);
  group_sync(tp, bar);
  if (tid == 0) {
    accepted_before += *accepted;
    *accepted = 0.0;
  }
  __syncwarp();  // the first warp saves the accumulators
  if (P.save && st) {
    for (int i = tid; i < N; i += tp) {
      const int x = i % L, y = i / L;
      st_spins[((x + y) & 1) * NH + (i >> 1)] = static_cast<int8_t>(spin_at(x, y));
    }
    if (tid < kAccDoubles) reinterpret_cast<double*>(st)[tid] = meter.acc[tid];
  }
  meter.write_record(P.records + (sy.rec_offset + path) * MP_NREC, 0, 0.0, P.s_end,
                     n_meas_done, N, tp, bar, accepted_before,
                     (P.save && st) ? reinterpret_cast<double*>(st) + kAccDoubles : nullptr);
  if (P.spins != nullptr) {
    double* out = P.spins + P.spin_offset[sys_idx] + path * 3 * static_cast<int64_t>(N);
    for (int i = tid; i < N; i += tp) {
      const int x = i % L, y = i / L;
      out[3 * i + 0] = 0.0;
      out[3 * i + 1] = 0.0;
      out[3 * i + 2] = static_cast<double>(spin_at(x, y));
    }
  }
  group_sync(tp, bar);  // the slice is reused by the next item
}

__global__ void __launch_bounds__(kIsingThreads, 1) ising_kernel(const SweepParams P) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int s_item;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) s_item = atomicAdd(P.queue, 1);
    __syncthreads();
    const int item = s_item;
    if (item >= P.n_items) return;
    const WorkItem it = P.items[item];
    const DevSystem sy = P.systems[it.sys];
    const int g = static_cast<int>(threadIdx.x) / sy.tp;
    const int tid = static_cast<int>(threadIdx.x) - g * sy.tp;
    if (g < it.count) run_path_ising(sy, it.sys, it.path0 + g, P, smem + g * sy.slice_bytes, tid, sy.tp, 1 + g);
  }
}

}  // namespace

// Threads per path of an L x L lattice when the caller names none: the count
// whose strips fill its lanes best, weighed with the warps an SM then holds (of
// 32; 13 reach 0.56, 26 0.94 of the rate, at L = 128) and with the barrier that
// more than one warp per path needs (about 7%).  Attempts/s by threads per path:
// L = 60 32: 9.9e11, 64: 9.0e11, 256: 6.0e11; L = 100 32: 7.7e11, 64: 9.0e11, 128:
// 9.2e11; L = 128 32: 6.4e11, 64: 9.8e11, 128: 1.02e12.
// `full`: for a GPU full of paths; `loaded`: for paths_per_sm, at most `most`.  (In one
// pass: the segment search takes some 10 us of a small call.)
IsingThreads ising_threads(int L, int64_t paths_per_sm, int smem_max, int ring, int most) {
  const int S = (L / 2) * ((L + 3) / 4);
  double best_full = -1.0, best_loaded = -1.0;
  IsingThreads best{32, 32};
  for (int t = 32; t <= kIsingThreads && (t == 32 || t < 2 * S); t += 32) {
    const int slice = (slice_spin_offset(t, ring, kRedBytes) + ising_slice_spin_bytes(L) + 127) / 128 * 128;
    const int64_t fit = std::min<int64_t>(smem_max / slice, t > 32 ? std::min(15, kIsingThreads / t) : kIsingThreads / t);
    if (fit < 1) continue;
    const int q = ising_segment(L, t), units = (L / 2) * (((L + 3) / 4 + q - 1) / q);
    const double fill = S / (static_cast<double>(t) * ((units + t - 1) / t) * (q + 0.4));
    auto rate = [&](int64_t paths) {
      return fill * std::pow(std::min(1.0, static_cast<double>(std::min(fit, paths)) * t / 1024.0), 0.65) *
             (t == 32 ? 1.0 : 0.93);
    };
    const double full = rate(fit), loaded = rate(paths_per_sm);
    if (full > best_full + 1e-9) {
      best_full = full;
      best.full = t;
    }
    if (t <= most && loaded > best_loaded + 1e-9) {
      best_loaded = loaded;
      best.loaded = t;
    }
  }
  return best;
}

cudaError_t ising_prepare(int device, int* max_dynamic, int* max_threads) {
  int optin = 0;
  cudaError_t e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
  if (e != cudaSuccess) return e;
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, ising_kernel);
  if (e != cudaSuccess) return e;
  *max_dynamic = optin - static_cast<int>(fa.sharedSizeBytes);
  *max_threads = fa.maxThreadsPerBlock;
  return cudaFuncSetAttribute(ising_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, *max_dynamic);
}

cudaError_t ising_occupancy(int cta, int smem, int* blocks) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, ising_kernel, cta, smem);
}

cudaError_t launch_ising(const SweepParams& p, int grid, int cta, int smem, cudaStream_t st) {
  ising_kernel<<<grid, cta, smem, st>>>(p);
  return cudaGetLastError();
}

}  // namespace mpk
