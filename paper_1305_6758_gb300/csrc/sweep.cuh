// Shared-memory checkerboard sweep of many independent simulation paths.
//
// What one path computes (Sec. 2.2 of Rakic et al.): a random initial state,
// then n_therm + n_meas lattice sweeps of Metropolis single spin-flip updates
// of the Heisenberg energy, Eq. (1) plus a Zeeman term -h sum S^z, with unit
// spins of Eq. (2); after every measurement sweep the per-site energy and
// total spin enter FP64 running sums, and the path's outputs are their means
// plus the final state.
//
// GB300 mapping: every path's lattice lives in shared memory for the whole
// run (no HBM traffic per sweep).  A persistent CTA pulls work items from an
// atomic queue; an item is `count` paths of one system, each run by its own
// group of `tp` threads with its own named barrier.  A sweep is two
// half-sweeps: all sites of colour (x+y+z) mod 2 = 0, then all of colour 1.
// Sites of one colour have neighbours only of the other colour, so they
// update independently (this replaces the paper's N randomly chosen sites by
// the checkerboard order; both leave the Boltzmann distribution invariant).
// The colour-1 pass sees final colour-0 neighbours, so the sum over colour-1
// sites of S_i . h_loc,i visits every bond once: the energy comes for free.
//
// Shared-memory layout of one path: [colour][(x, y) pairs | z][half index],
// the half index of site i = x + L(y + Lz) being i >> 1, so a spin is one
// 8-byte and one 4-byte load (16 + 8 in FP64) and a warp's 32 consecutive
// sites of one colour and their +-y, +-z neighbours are consecutive elements.
#pragma once
#include <cstdint>
#include <type_traits>

#include "common.cuh"
#include "fixed64.cuh"
#include "philox.cuh"

namespace mpk {

// ------------------------------------------------------------ arithmetic --
template <typename Real>
struct Arith;

// FP32 form: 23-bit uniforms (exact in float, open interval), hardware
// approximations for rsqrt, sin/cos and 2^x.  |S'| = 1 to about 1e-6.
template <>
struct Arith<float> {
  // 1 + m 2^-23 with m the top 23 bits of r, built from the bits (no int->float
  // conversion; the sum is one shift-and-add instruction, an "or" would be
  // two); the uniform is that minus (1 - 2^-24) = (2m + 1) 2^-24, exactly.
  static __device__ __forceinline__ float one_plus(uint32_t r) {
    return __uint_as_float(0x3f800000u + (r >> 9));
  }
  static __device__ __forceinline__ float uni(uint32_t r) { return one_plus(r) - 0.99999994f; }
  // Trial direction uniform on the sphere: cos(theta) = 2u0 - 1, phi = 2 pi u1.
  static __device__ __forceinline__ void trial(uint32_t r0, uint32_t r1, float& x, float& y,
                                               float& z) {
    z = fmaf(2.0f, uni(r0), -1.0f);  // 2 u0 - 1, exact, never +-1
    const float q = fmaf(-z, z, 1.0f);  // 1 - z^2 > 0
    const float rad = q * rsqrtf(q);
    float s, c;
    // phi - pi = 2 pi (u1 - 1/2) lies in (-pi, pi), where the hardware sin/cos
    // are accurate; cos(phi) = -cos(phi - pi), sin(phi) = -sin(phi - pi).
    __sincosf(fmaf(6.28318531f, one_plus(r1), -9.42477763f), &s, &c);
    x = __fmul_rn(-rad, c);
    y = __fmul_rn(-rad, s);
  }
  static __device__ __forceinline__ void init_angles(uint32_t r0, uint32_t r1, float& x, float& y,
                                                     float& z) {
    float st, ct, sp, cp;
    sincospif(uni(r0), &st, &ct);
    sincospif(2.0f * uni(r1), &sp, &cp);
    x = st * cp;
    y = st * sp;
    z = ct;
  }
  // a.b, every rounding spelled out: where a sum of products is left to the
  // compiler, which product it rounds first changes with the code around it,
  // and with it one accept decision in 1e8.
  static __device__ __forceinline__ float dot(float ax, float ay, float az, float bx, float by, float bz) {
    return __fmaf_rn(az, bz, __fmaf_rn(ax, bx, __fmul_rn(ay, by)));
  }
  static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
  static __device__ __forceinline__ float square(float x, float y, float z) {
    return __fadd_rn(__fmaf_rn(y, y, __fmul_rn(x, x)), __fmul_rn(z, z));
  }
  static __device__ __forceinline__ float square_pair(float x, float y, float z) {
    return __fadd_rn(__fmaf_rn(x, x, __fmul_rn(y, y)), __fmul_rn(z, z));
  }
  // Metropolis test of the move S -> S + d in the local field (hx, hy, hz):
  // accept when dE <= 0, else iff u < exp(-beta dE) = 2^(-x), with
  // x = beta log2(e) dE = (-b J) d.h_loc + (-b h) d_z and b = beta log2(e)
  // precomputed per path (the two products are loop invariants).  One compare
  // decides both: 2^(-x) >= 1 > u for x <= 0 (the hardware's ex2 gives at least 1
  // for every argument >= 0, checked over all floats).
  static __device__ __forceinline__ bool accept_move(float dx, float dy, float dz, float hx,
                                                     float hy, float hz, float J, float hf,
                                                     float blog2e, uint32_t r2) {
    const float x = __fmaf_rn(__fmul_rn(-blog2e, J), dot(dx, dy, dz, hx, hy, hz), __fmul_rn(__fmul_rn(-blog2e, hf), dz));
    float p;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(p) : "f"(-x));
    return uni(r2) < p;
  }
  static __device__ __forceinline__ float beta_param(double beta) {
    return static_cast<float>(beta * 1.4426950408889634);
  }
  static __device__ __forceinline__ float shfl(float v, int o) {
    return __shfl_xor_sync(0xffffffffu, v, o);
  }
};

// FP64 form: 32-bit uniforms (r + 1/2) 2^-32.  Trial spins are fix_trial's
// (fixed64.cuh); where the FP32 stage does not decide a move, the local-field dot
// product is rounded term by term in the order ((dx hx + dy hy) + dz hz) with no
// fused multiply-add and the Boltzmann factor is the library's exp, so that dE is a
// plain FP64 evaluation's of the same spins.
template <>
struct Arith<double> {
  static __device__ __forceinline__ double uni(uint32_t r) {
    return (static_cast<double>(r) + 0.5) * 0x1p-32;
  }
  static __device__ __forceinline__ void init_angles(uint32_t r0, uint32_t r1, double& x,
                                                     double& y, double& z) {
    const double th = __dmul_rn(3.141592653589793, uni(r0));
    const double ph = __dmul_rn(2.0 * 3.141592653589793, uni(r1));
    double st, ct, sp, cp;
    sincos(th, &st, &ct);
    sincos(ph, &sp, &cp);
    x = __dmul_rn(st, cp);
    y = __dmul_rn(st, sp);
    z = ct;
  }
  static __device__ __forceinline__ double square(double x, double y, double z) {
    return fma(z, z, fma(y, y, x * x));
  }
  static __device__ __forceinline__ double delta_e(double dx, double dy, double dz, double hx,
                                                   double hy, double hz, double J, double hf) {
    const double dot = __dadd_rn(__dadd_rn(__dmul_rn(dx, hx), __dmul_rn(dy, hy)), __dmul_rn(dz, hz));
    return __dsub_rn(__dmul_rn(-J, dot), __dmul_rn(hf, dz));
  }
  static __device__ __forceinline__ bool accept_move(double dx, double dy, double dz, double hx,
                                                     double hy, double hz, double J, double hf,
                                                     double beta, uint32_t r2) {
    const double dE = delta_e(dx, dy, dz, hx, hy, hz, J, hf);
    return dE <= 0.0 || uni(r2) < exp(__dmul_rn(-beta, dE));
  }
  static __device__ __forceinline__ double shfl(double v, int o) {
    return __shfl_xor_sync(0xffffffffu, v, o);
  }
};

// -------------------------------------------------------------- geometry --
// Periodic simple cubic lattice with compile-time L (even).  site() returns
// the site index of half index h in colour c and fills the half indices of
// its neighbours in the other colour, in the fixed order +x, -x, +y, -y, +z, -z.
// Half index h = hx + HL*y + HP*z with hx = x / 2.  kMixed: the geometry as
// run by the mixed-size kernel (which takes the column-walk chunks of
// column_chunk_fp32(L, true)).
template <int L, bool kMixed = false>
struct GeomSC {
  static constexpr bool kInMixed = kMixed;
  static constexpr int N = L * L * L;
  static constexpr int NH = N / 2;
  static constexpr int HL = L / 2;
  static constexpr int HP = L * L / 2;
  static constexpr int NNB = 6;
  static constexpr bool kColumns = true;
  __device__ __forceinline__ int count(int) const { return NH; }
  static __device__ __forceinline__ constexpr int stride() { return NH; }
  __device__ __forceinline__ int site(int h, int c, int* nb, int& nn) const {
    const int hx = h % HL;
    const int t = h / HL;
    const int y = t % L;
    const int z = t / L;
    const int p = (y + z + c) & 1;
    const int x = 2 * hx + p;
    const int hrow = h - hx;
    nb[0] = hrow + ((x + 1 == L) ? 0 : ((x + 1) >> 1));
    nb[1] = hrow + ((x == 0) ? ((L - 1) >> 1) : ((x - 1) >> 1));
    nb[2] = (y == L - 1) ? h - (L - 1) * HL : h + HL;
    nb[3] = (y == 0) ? h + (L - 1) * HL : h - HL;
    nb[4] = (z == L - 1) ? h - (L - 1) * HP : h + HP;
    nb[5] = (z == 0) ? h + (L - 1) * HP : h - HP;
    nn = 6;
    return 2 * h + p;
  }
};

// Periodic simple cubic lattice of run-time L (even), every site decoded from
// its half index (neighbours in the same fixed order as GeomSC): the geometry
// of lattices updated in place in HBM, which are too large for a ring of
// half-planes in shared memory.
struct GeomSCDyn {
  int L;
  static constexpr int NNB = 6;
  static constexpr bool kColumns = false;
  __device__ __forceinline__ int count(int) const { return L * L * L / 2; }
  __device__ __forceinline__ int stride() const { return L * L * L / 2; }
  __device__ __forceinline__ int site(int h, int c, int* nb, int& nn) const {
    const int HL = L / 2, HP = L * L / 2;
    const int hx = h % HL;
    const int t = h / HL;
    const int y = t % L;
    const int z = t / L;
    const int p = (y + z + c) & 1;
    const int x = 2 * hx + p;
    const int hrow = h - hx;
    nb[0] = hrow + ((x + 1 == L) ? 0 : ((x + 1) >> 1));
    nb[1] = hrow + ((x == 0) ? ((L - 1) >> 1) : ((x - 1) >> 1));
    nb[2] = (y == L - 1) ? h - (L - 1) * HL : h + HL;
    nb[3] = (y == 0) ? h + (L - 1) * HL : h - HL;
    nb[4] = (z == L - 1) ? h - (L - 1) * HP : h + HP;
    nb[5] = (z == 0) ? h + (L - 1) * HP : h - HP;
    nn = 6;
    return 2 * h + p;
  }
};

// Open chain of N spins: colour i mod 2, neighbours i-1 then i+1 where they exist.
struct GeomChain {
  int N;
  static constexpr int NNB = 2;
  static constexpr bool kColumns = false;
  static constexpr int HP = 1;
  __device__ __forceinline__ int count(int c) const { return c == 0 ? (N + 1) >> 1 : N >> 1; }
  // even, so that every (x, y) pair array starts on a pair boundary
  __device__ __forceinline__ int stride() const { return (((N + 1) >> 1) + 1) & ~1; }
  __device__ __forceinline__ int site(int h, int c, int* nb, int& nn) const {
    const int i = 2 * h + c;
    nn = 0;
    if (i > 0) nb[nn++] = (i - 1) >> 1;
    if (i < N - 1) nb[nn++] = (i + 1) >> 1;
    return i;
  }
};

// ----------------------------------------------------------- group sync --
// tp threads of one path synchronise on their own named barrier (1 + group),
// or with __syncwarp when the path is one warp.
__device__ __forceinline__ void group_sync(int tp, int bar) {
  if (tp == 32) {
    __syncwarp();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(tp) : "memory");
  }
}

// ------------------------------------------------------- one attempt -----
// A 96-bit integer sum.
struct Wide {
  uint32_t w0 = 0, w1 = 0, w2 = 0;
  __device__ __forceinline__ void add(uint32_t a, uint32_t b, uint32_t c) {
    asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
        : "+r"(w0), "+r"(w1), "+r"(w2)
        : "r"(a), "r"(b), "r"(c));
  }
  __device__ __forceinline__ void add(int64_t v) {
    const uint32_t hi = static_cast<uint32_t>(static_cast<uint64_t>(v) >> 32);
    add(static_cast<uint32_t>(v), hi, static_cast<uint32_t>(static_cast<int32_t>(hi) >> 31));
  }
  __device__ __forceinline__ void add_warp() {  // every lane gets the warp's sum
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const uint32_t a = __shfl_xor_sync(0xffffffffu, w0, o), b = __shfl_xor_sync(0xffffffffu, w1, o),
                     c = __shfl_xor_sync(0xffffffffu, w2, o);
      add(a, b, c);
    }
  }
  // The value in units of 2^-unit as a double (the scale goes into the exponent).
  __device__ __forceinline__ double real(int unit) const {
    const double d = real();
    const int hi = __double2hiint(d);
    return hi == 0 ? 0.0 : __hiloint2double(hi - (unit << 20), __double2loint(d));
  }
  // The value as a double.
  __device__ __forceinline__ double real() const {
    const int64_t low = static_cast<int64_t>((static_cast<uint64_t>(w1) << 32) | w0);
    const int32_t top = static_cast<int32_t>(w2) - static_cast<int32_t>(low >> 63);  // 0 if 64 bits hold it
    double d = static_cast<double>(low);
    if (top != 0) d = fma(static_cast<double>(top), 0x1p64, d);
    return d;
  }
};

// Sums of four values over the warp: lane l gets that of value (l & 3), in the
// order a, c, b, d.  Two exchanges halve what a lane carries, so 18 words are
// shuffled instead of the 60 of four butterflies.
__device__ __forceinline__ Wide warp_sums(const Wide& a, const Wide& b, const Wide& c, const Wide& d, int lane) {
  auto pick = [](bool second, const Wide& x, const Wide& y) {
    Wide r;
    r.w0 = second ? y.w0 : x.w0;
    r.w1 = second ? y.w1 : x.w1;
    r.w2 = second ? y.w2 : x.w2;
    return r;
  };
  auto from = [](const Wide& x, int o) {
    Wide r;
    r.w0 = __shfl_xor_sync(0xffffffffu, x.w0, o);
    r.w1 = __shfl_xor_sync(0xffffffffu, x.w1, o);
    r.w2 = __shfl_xor_sync(0xffffffffu, x.w2, o);
    return r;
  };
  const bool odd = lane & 1, high = lane & 2;
  Wide x = pick(odd, a, c), y = pick(odd, b, d);  // even lanes a, b; odd lanes c, d
  const Wide xs = from(pick(odd, c, a), 1), ys = from(pick(odd, d, b), 1);
  x.add(xs.w0, xs.w1, xs.w2);
  y.add(ys.w0, ys.w1, ys.w2);
  Wide z = pick(high, x, y);
  const Wide zs = from(pick(high, y, x), 2);
  z.add(zs.w0, zs.w1, zs.w2);
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    const Wide t = from(z, o);
    z.add(t.w0, t.w1, t.w2);
  }
  return z;
}

// Per-thread partial sums of the measurement of one sweep: sums of S . h over
// the colour-1 sites and of the new spins.  FP64 form: exact integers, the
// spins in units of 2^-53 and S . h in units of 2^-57.
template <typename Real>
struct Partials {
  Real eb{}, mx{}, my{}, mz{};
};
template <>
struct Partials<double> {
  Wide eb, mx, my, mz;
};
constexpr int kEnergyBits = 57;
constexpr double kEnergyUnit = 0x1p-57, kSpinUnit = 0x1p-53;

// ------------------------------------------------------------ spin views --
// A spin component as the kernels store it: float, or (FP64 form) the 64-bit
// integer of fixed64.cuh.  Saved states and read-out spins are doubles.
template <typename Real>
struct Stored;
template <>
struct Stored<float> {
  using C = float;
  using P2 = float2;
  static __device__ __forceinline__ C from(float v) { return v; }
  static __device__ __forceinline__ float real(C v) { return v; }
};
template <>
struct Stored<double> {
  using C = int64_t;
  using P2 = longlong2;
  static __device__ __forceinline__ C from(double v) { return __double2ll_rn(v * 0x1p53); }
  static __device__ __forceinline__ double real(C v) { return static_cast<double>(v) * kSpinUnit; }
};

template <typename Real>
struct V3 {
  typename Stored<Real>::C x, y, z;
};
template <typename Real>
__device__ __forceinline__ V3<Real> add3(V3<Real> a, V3<Real> b) {
  return V3<Real>{a.x + b.x, a.y + b.y, a.z + b.z};
}

// S spins of one colour (or one half-plane): their (x, y) pairs, then their z
// components.  base must be aligned to a pair and S even.
template <typename Real>
struct SpinView {
  using C = typename Stored<Real>::C;
  using P2 = typename Stored<Real>::P2;
  P2* xy;
  C* z;
  __device__ __forceinline__ SpinView(Real* base, int S)
      : xy(reinterpret_cast<P2*>(base)), z(reinterpret_cast<C*>(base) + 2 * S) {}
  __device__ __forceinline__ V3<Real> ld(int h) const {
    const P2 v = xy[h];
    return V3<Real>{v.x, v.y, z[h]};
  }
  __device__ __forceinline__ void st(int h, C a, C b, C c) const {
    P2 v;
    v.x = a;
    v.y = b;
    xy[h] = v;
    z[h] = c;
  }
};

// | |S| - 1 | of a stored spin.
__device__ __forceinline__ float norm_error(V3<float> v) {
  return fabs(sqrt(v.x * v.x + v.y * v.y + v.z * v.z) - 1.0f);
}
__device__ __forceinline__ double norm_error(V3<double> v) {
  // |S|^2 - 1 in units of 2^-60 from the high halves of the squares; for a
  // unit spin |S| - 1 is half of it (one FP64 square root costs 570 cycles)
  const int64_t a = v.x << 9, b = v.y << 9, c = v.z << 9;
  const int64_t d = __mul64hi(a, a) + __mul64hi(b, b) + __mul64hi(c, c) - (int64_t{1} << 60);
  const double t = static_cast<double>(d < 0 ? -d : d) * 0x1p-61;
  if (t < 0x1p-30) return t;
  const double x = Stored<double>::real(v.x), y = Stored<double>::real(v.y), z = Stored<double>::real(v.z);
  return fabs(sqrt(x * x + y * y + z * z) - 1.0);  // a restored state that holds no unit spin
}

// --------------------------------------------------------- sine table ----
// The table of fix_trial in the CTA's shared memory (FP64 kernels).
static __device__ const SineTable kSineTable = make_sine_table();
__device__ __forceinline__ uint64_t* sine_shared() {
  __shared__ uint64_t t[256];
  return t;
}

// ------------------------------------------------------------ couplings --
// What the accept test of a path needs of its system.
template <typename Real>
struct Couplings;
template <>
struct Couplings<float> {
  float J, hf, bp;
  __device__ explicit Couplings(const DevSystem* s)
      : J(static_cast<float>(s->J)), hf(static_cast<float>(s->h)), bp(Arith<float>::beta_param(s->beta)) {}
};
template <>
struct Couplings<double> {
  const DevSystem* sys;
  float cj, ch;    // log2 of the acceptance is cj d.h + ch d_z, d and h in units of 2^-28
  float lo, hi;    // 1 -+ the bound on the relative error of the FP32 acceptance (0 and infinity: none)
  __device__ explicit Couplings(const DevSystem* s) : sys(s) {
    const double bj = s->beta * s->J, bh = s->beta * s->h;
    cj = static_cast<float>(bj * 1.4426950408889634 * 0x1p-56);
    ch = static_cast<float>(bh * 1.4426950408889634 * 0x1p-28);
    // Bound: |d| <= 2, |h| <= 6; a trial component is off by at most 1.2e-6
    // (2^-21.2 of the hardware sine and cosine, 2^-23 of their argument, 2^-22
    // of the radius), d by 1.5e-6, h by 3.7e-7, so d.h by 1.9e-5; the exponent's
    // own roundings are 2^-21 of at most 33 (beyond that the test is decided),
    // ex2 and the uniform add 2^-22.  Taken a third larger, which covers
    // exp(+-bound) - 1, the error of the acceptance, while it is below 1/4.  Beyond
    // that (beta |J| = 1e4) no move is decided here: nothing is below 0, and
    // nothing above p times infinity (a p of 0 makes it NaN).
    const float tol = static_cast<float>(2.5e-5 * fabs(bj) + 3e-6 * fabs(bh) + 2e-5);
    lo = tol < 0.25f ? 1.0f - tol : 0.0f;
    hi = tol < 0.25f ? 1.0f + tol : __int_as_float(0x7f800000);
  }
};

// The Metropolis step at site i (half index hh of the colour view `own`)
// given its local field f, Sec. 2.2: trial spin, energy change from the local
// field, acceptance test.
//
// settle: the trial spin t and the spin a held at the site are known; act =
// false (a thread that walks along without a site) changes and counts
// nothing.
template <bool kMeas, bool kEnergy>
__device__ __forceinline__ void settle(V3<float> t, uint32_t r2, const SpinView<float>& own, int hh, V3<float> a,
                                       V3<float> f, const Couplings<float>& cp, bool act, int& accepted,
                                       Partials<float>& part) {
  using A = Arith<float>;
  float nx = a.x, ny = a.y, nz = a.z;
  if (A::accept_move(A::sub(t.x, a.x), A::sub(t.y, a.y), A::sub(t.z, a.z), f.x, f.y, f.z, cp.J, cp.hf, cp.bp, r2) &&
      act) {
    own.st(hh, t.x, t.y, t.z);
    nx = t.x;
    ny = t.y;
    nz = t.z;
    ++accepted;
  }
  if (kMeas) {
    part.mx += act ? nx : 0.0f;
    part.my += act ? ny : 0.0f;
    part.mz += act ? nz : 0.0f;
    if (kEnergy) {
      const float b = A::dot(nx, ny, nz, f.x, f.y, f.z);
      part.eb += act ? b : 0.0f;
    }
  }
}
template <bool kMeas, bool kEnergy>
__device__ __forceinline__ void update_spin(uint32_t i, const PhiloxPrefix& pre, const PhiloxKeys& key,
                                            const SpinView<float>& own, int hh, V3<float> a, V3<float> f,
                                            const Couplings<float>& cp, bool act, int& accepted,
                                            Partials<float>& part) {
  const Philox4 r = philox4x32_10(i, pre, key);
  V3<float> t;
  Arith<float>::trial(r.x, r.y, t.x, t.y, t.z);
  settle<kMeas, kEnergy>(t, r.z, own, hh, a, f, cp, act, accepted, part);
}
template <bool kMeas, bool kEnergy>
__device__ __forceinline__ void update(uint32_t i, const PhiloxPrefix& pre, const PhiloxKeys& key,
                                       const SpinView<float>& own, int hh, V3<float> f,
                                       const Couplings<float>& cp, int& accepted, Partials<float>& part) {
  update_spin<kMeas, kEnergy>(i, pre, key, own, hh, own.ld(hh), f, cp, true, accepted, part);
}

// The accept test in FP64, for moves whose FP32 acceptance is too close to
// the uniform to decide: d and h in units of 2^-53.
static __device__ __noinline__ bool accept_exact(int64_t dx, int64_t dy, int64_t dz, int64_t hx, int64_t hy, int64_t hz,
                                          const DevSystem* sys, uint32_t r2) {
  using A = Arith<double>;
  using S = Stored<double>;
  return A::accept_move(S::real(dx), S::real(dy), S::real(dz), S::real(hx), S::real(hy), S::real(hz), sys->J,
                        sys->h, sys->beta, r2);
}

// FP64 form.  What bounds it is FP64 issue (76 cycles per warp instruction
// and scheduler), so none is left on the common path: the local field is an
// integer sum, the accept test u < exp(-beta dE) is decided in FP32 wherever u
// lies outside the FP32 acceptance's error bound (all but about 1e-5 of the
// moves; those take accept_exact), and the trial spin is evaluated to 2^-53 in
// integers (fix_trial), by warps in which a move was accepted.  L = 16, three
// temperatures of 1024 paths: 5.2e9 attempts/s with FP64 arithmetic, 7.1e10 so in
// thermalisation and 6.1e10 in measured sweeps.
//
// The FP32 stage of a move: the trial direction in units of 2^-28 and the uniform.
struct FixDraw {
  float tx, ty, tz, u;
};
__device__ __forceinline__ FixDraw fix_draw(const Philox4& r, const FixRoot& q) {
  const float rad = q.nf * q.y * 0x1p-4f;  // sqrt(n) 2^-32 2^28
  float s, c;
  // phi - pi = (r1 + 1/2 - 2^31) 2 pi 2^-32; sine and cosine change sign
  __sincosf(static_cast<float>(static_cast<int32_t>(r.y ^ 0x80000000u)) * 1.46291808e-9f, &s, &c);
  return FixDraw{-rad * c, -rad * s, static_cast<float>(static_cast<int32_t>(r.x ^ 0x80000000u)) * 0.125f,
                 fmaf(static_cast<float>(r.z), 0x1p-32f, 0x1p-33f)};
}
// Accepted for certain (ok), or undecided (open; NaN and infinity included).
__device__ __forceinline__ void fix_test(const FixDraw& d, V3<double> a, V3<double> f, const Couplings<double>& cp,
                                         bool& ok, bool& open) {
  auto f28 = [](int64_t v) { return static_cast<float>(static_cast<int32_t>(v >> 25)); };
  const float dx = d.tx - f28(a.x), dy = d.ty - f28(a.y), dz = d.tz - f28(a.z);
  const float dot = dx * f28(f.x) + dy * f28(f.y) + dz * f28(f.z);
  float p;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(p) : "f"(fmaf(cp.cj, dot, cp.ch * dz)));
  ok = d.u < p * cp.lo;
  open = !ok && !(d.u > p * cp.hi);
}

// The move drawn by r at the spin a in the local field f: accepted(trial spin)
// is called when it is accepted (within the branch that evaluates the trial
// spin: a second branch on the outcome costs 15%).
template <class F>
__device__ __forceinline__ void move_fixed(const Philox4& r, V3<double> a, V3<double> f, const Couplings<double>& cp,
                                           F&& accepted) {
  const FixRoot q = fix_root(r.x);
  bool ok, open;
  fix_test(fix_draw(r, q), a, f, cp, ok, open);
  if (ok || open) {
    const Fix3 t = fix_trial(r.x, r.y, q, sine_shared());
    if (open) ok = accept_exact(t.x - a.x, t.y - a.y, t.z - a.z, f.x, f.y, f.z, cp.sys, r.z);
    if (ok) accepted(V3<double>{t.x, t.y, t.z});
  }
}

// S . h in units of 2^-57, from (S 2^62) (h 2^59) 2^-64.
__device__ __forceinline__ int64_t spin_dot(V3<double> s, V3<double> h) {
  return __mul64hi(s.x << 9, h.x << 6) + __mul64hi(s.y << 9, h.y << 6) + __mul64hi(s.z << 9, h.z << 6);
}

template <bool kMeas, bool kEnergy>
__device__ __forceinline__ void update(uint32_t i, const PhiloxPrefix& pre, const PhiloxKeys& key,
                                       const SpinView<double>& own, int hh, V3<double> f,
                                       const Couplings<double>& cp, int& accepted, Partials<double>& part) {
  const Philox4 r = philox4x32_10(i, pre, key);
  const V3<double> a = own.ld(hh);
  V3<double> n = a;
  move_fixed(r, a, f, cp, [&](V3<double> t) {
    own.st(hh, t.x, t.y, t.z);
    n = t;
    ++accepted;
  });
  if (kMeas) {
    part.mx.add(n.x);
    part.my.add(n.y);
    part.mz.add(n.z);
    if (kEnergy) part.eb.add(spin_dot(n, f));
  }
}

// One-site form (see run_path): a move drawn ahead of its update.  A thread
// without a site (act = false) reads no spin of the colour that the others are
// writing.
template <typename Real>
struct Ahead;
template <>
struct Ahead<float> {
  V3<float> t;
  uint32_t r2;
  __device__ __forceinline__ explicit Ahead(const Philox4& r) : r2(r.z) { Arith<float>::trial(r.x, r.y, t.x, t.y, t.z); }
  template <bool kMeas, bool kEnergy>
  __device__ __forceinline__ void apply(const SpinView<float>& own, int hh, V3<float> f, const Couplings<float>& cp,
                                        bool act, int& accepted, Partials<float>& part) const {
    V3<float> a{};
    if (act) a = own.ld(hh);
    settle<kMeas, kEnergy>(t, r2, own, hh, a, f, cp, act, accepted, part);
  }
};
template <>
struct Ahead<double> {
  FixDraw d;
  Fix3 t;
  uint32_t r2;
  __device__ __forceinline__ explicit Ahead(const Philox4& r) : r2(r.z) {
    const FixRoot q = fix_root(r.x);
    d = fix_draw(r, q);
    t = fix_trial(r.x, r.y, q, sine_shared());
  }
  template <bool kMeas, bool kEnergy>
  __device__ __forceinline__ void apply(const SpinView<double>& own, int hh, V3<double> f, const Couplings<double>& cp,
                                        bool act, int& accepted, Partials<double>& part) const {
    V3<double> a{};
    if (act) a = own.ld(hh);
    bool ok, open;
    fix_test(d, a, f, cp, ok, open);
    if (open && act) ok = accept_exact(t.x - a.x, t.y - a.y, t.z - a.z, f.x, f.y, f.z, cp.sys, r2);
    ok = ok && act;
    const V3<double> n = ok ? V3<double>{t.x, t.y, t.z} : a;
    if (ok) {
      own.st(hh, n.x, n.y, n.z);
      ++accepted;
    }
    if (kMeas && act) {
      part.mx.add(n.x);
      part.my.add(n.y);
      part.mz.add(n.z);
      if (kEnergy) part.eb.add(spin_dot(n, f));
    }
  }
};

// One Metropolis attempt with the neighbours' half indices nb[0..nn) in `oth`,
// summed in the fixed order nb[0], nb[1], ...
template <typename Real, int NNB, bool kMeas, bool kEnergy>
__device__ __forceinline__ void attempt(uint32_t i, const PhiloxPrefix& pre, const PhiloxKeys& key, const SpinView<Real>& own,
                                        const SpinView<Real>& oth, int hh, const int* nb, int nn,
                                        const Couplings<Real>& cp, int& accepted,
                                        Partials<Real>& part) {
  V3<Real> f{};
#pragma unroll
  for (int j = 0; j < NNB; ++j) {
    if (j < nn) f = add3(f, oth.ld(nb[j]));
  }
  update<kMeas, kEnergy>(i, pre, key, own, hh, f, cp, accepted, part);
}

// The column chunk U of a geometry (column_chunk in common.cuh).
template <typename Real, class Geom>
constexpr int kColumnChunk = column_chunk(static_cast<int>(sizeof(Real)), 2 * Geom::HL, Geom::kInMixed);

// One half-sweep of one thread: every site of colour c it owns.
//
// Column-segment walk (simple cubic, K > 0): a colour's sites form L^2/2
// columns col = x/2 + (L/2) y of L planes each (half index col + (L^2/2) z);
// each column is cut into K segments of L/K planes, and the HP * K units
// (column col, segment g), numbered u = g * HP + col, are dealt out to the
// threads round by round (thread tid takes u = tid, tid + tp, ...), so the
// lanes of a warp work on consecutive columns of the same planes and their
// shared-memory accesses are consecutive elements.  A segment is walked in
// chunks of kColumnChunk planes whose sites the compiler interleaves.  Within a segment the +-x
// and +-y neighbour offsets are fixed, and since the x parity flips from
// plane to plane, the other colour's spin at the site's own half index is
// both an x neighbour of the site in plane z and the -z neighbour of the site
// in plane z + 1, while the +z neighbour of one site is an x neighbour of the
// next: after the first site of a segment two of the six neighbours are
// already in registers.  The two x neighbours are added first, in either
// order (a + b = b + a exactly), so the sum keeps the fixed order +x, -x, +y,
// -y, +z, -z.  K = 0: every site decoded from its half index (open chains).
template <typename Real, class Geom, bool kMeas, bool kEnergy>
__device__ __forceinline__ void half_sweep(const Geom& geo, int c, const PhiloxPrefix& pre,
                                           const PhiloxKeys& key, Real* sp, int tid,
                                           int tp, int K, const int4* units, const Couplings<Real>& cp,
                                           int& accepted, Partials<Real>& part) {
  const int S = geo.stride();
  const SpinView<Real> own(sp + c * 3 * S, S);
  const SpinView<Real> oth(sp + (1 - c) * 3 * S, S);
  if constexpr (Geom::kColumns) {
    if (K > 0) {
      constexpr int HL = Geom::HL, HP = Geom::HP, LL = 2 * Geom::HL;
      const int seg = LL / K;  // planes per segment
      constexpr int U = kColumnChunk<Real, Geom>;
      constexpr int NH = HP * LL;
      // Where chunks of two give a warp too few independent random-number
      // chains, the rounds of a thermalisation sweep are taken two at a time (u
      // and u + tp side by side; measurement sweeps keep the order of their FP32
      // sums, and FP64 has no registers for it: a third slower at L = 16).
      // Attempts/s before -> after, sweeps of all kinds: L = 10, 1000 paths (7
      // warps per SM) 1.36e11 -> 1.47e11, a full GPU 2.08e11 ->
      // 2.15e11, L = 22 1.71e11 -> 1.72e11, L = 26 1.73e11 -> 1.85e11.  Chunks
      // of three lose by it (L = 6: 1.21e11 -> 1.18e11), four rounds at a time
      // lose everywhere.
      int u_first = tid;
      if constexpr (sizeof(Real) == 4 && !kMeas && U == 2 && !Geom::kInMixed) {
        const int n_units = HP * K, rounds = (n_units + tp - 1) / tp;
        struct Unit {
          int hh, oyp, oym, pa, oxa, oxb;
          bool act;
          V3<Real> o0, mz;
        };
        for (; u_first < rounds / 2 * 2 * tp; u_first += 2 * tp) {
          Unit unit[2];
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            Unit& w = unit[j];
            // the last round may lack a unit for this thread: it goes along
            // with its other one and changes nothing
            w.act = j == 0 || u_first + tp < n_units;
            const int u = u_first + (j == 1 && w.act ? tp : 0);
            const int4 d = units != nullptr ? __ldg(units + u) : column_unit(LL, K, u);
            w.hh = d.x & 0x7fffffff;
            w.pa = static_cast<int>(static_cast<unsigned>(d.x) >> 31) ^ c;
            const int xa = (d.y << 8) >> 24, xb = d.y >> 24;  // signed bytes 2 and 3
            w.oxa = c ? xb : xa;
            w.oxb = c ? xa : xb;
            w.oyp = d.z;
            w.oym = d.w;
            w.o0 = oth.ld(w.hh);
            w.mz = oth.ld(d.y & 0xffff);
          }
          for (int zc = 0; zc < seg; zc += U) {
#pragma unroll
            for (int k = 0; k < U; ++k) {
#pragma unroll
              for (int j = 0; j < 2; ++j) {
                Unit& w = unit[j];
                const int nxo = w.hh + ((k & 1) ? w.oxb : w.oxa);
                const int zn = (k == U - 1 && w.hh + HP >= NH) ? w.hh + HP - NH : w.hh + HP;
                const V3<Real> cz = oth.ld(zn);
                const V3<Real> f = add3(
                    add3(add3(add3(add3(w.o0, oth.ld(nxo)), oth.ld(w.hh + w.oyp)), oth.ld(w.hh + w.oym)), cz), w.mz);
                update_spin<false, false>(static_cast<uint32_t>(2 * w.hh + ((k & 1) ? w.pa ^ 1 : w.pa)), pre, key, own,
                                          w.hh, own.ld(w.hh), f, cp, w.act, accepted, part);
                w.mz = w.o0;
                w.o0 = cz;
                w.hh += HP;
              }
            }
          }
        }
      }
      for (int u = u_first; u < HP * K; u += tp) {
        // the unit: half index hh of its first site and of that site's -z
        // neighbour, +-y offsets, and the x parity p of the site: it flips
        // from plane to plane, so sites an even number of planes after the
        // chunk's first take (pa, oxa), the others (pb, oxb), and within a
        // chunk the choice is made at compile time
        int hh, mzi, oyp, oym, pa, oxa, oxb;
        if (units != nullptr) {  // from the host's table (column_unit)
          const int4 d = __ldg(units + u);
          hh = d.x & 0x7fffffff;
          pa = static_cast<int>(static_cast<unsigned>(d.x) >> 31) ^ c;
          mzi = d.y & 0xffff;
          const int xa = (d.y << 8) >> 24, xb = d.y >> 24;  // signed bytes 2 and 3
          oxa = c ? xb : xa;
          oxb = c ? xa : xb;
          oyp = d.z;
          oym = d.w;
        } else {
          // u >= 0: unsigned division by the compile-time HP and HL needs no
          // sign fix-up
          const unsigned uu = static_cast<unsigned>(u);
          const int g = static_cast<int>(uu / HP);
          const int col = static_cast<int>(uu % HP);
          const int z0 = g * seg;
          const int hx = static_cast<int>(static_cast<unsigned>(col) % HL);
          const int y = static_cast<int>(static_cast<unsigned>(col) / HL);
          oyp = (y == LL - 1) ? -(LL - 1) * HL : HL;
          oym = (y == 0) ? (LL - 1) * HL : -HL;
          const int oxp1 = (hx == HL - 1) ? -(HL - 1) : 1;  // +x offset when x is odd
          const int oxm0 = (hx == 0) ? (HL - 1) : -1;         // -x offset when x is even
          pa = (y + z0 + c) & 1;
          oxa = pa ? oxp1 : oxm0;
          oxb = pa ? oxm0 : oxp1;
          hh = col + HP * z0;
          mzi = z0 == 0 ? hh + (LL - 1) * HP : hh - HP;
        }
        int pb = pa ^ 1;
        const int oxx = oxa ^ oxb;
        V3<Real> o0 = oth.ld(hh);   // the other colour at the site's half index
        V3<Real> mz = oth.ld(mzi);  // -z neighbour
        for (int zc = 0; zc < seg; zc += U) {
#pragma unroll
          for (int k = 0; k < U; ++k, hh += HP) {
            const int p = (k & 1) ? pb : pa;
            const int nxo = hh + ((k & 1) ? oxb : oxa);
            // chunks start at multiples of U, which divides L: only a chunk's
            // last plane can be plane L - 1, whose +z neighbour wraps
            const int zn = (k == U - 1 && hh + HP >= NH) ? hh + HP - NH : hh + HP;
            const V3<Real> cz = oth.ld(zn);
            const V3<Real> f =
                add3(add3(add3(add3(add3(o0, oth.ld(nxo)), oth.ld(hh + oyp)), oth.ld(hh + oym)), cz), mz);
            update<kMeas, kEnergy>(static_cast<uint32_t>(2 * hh + p), pre, key, own, hh, f, cp, accepted, part);
            mz = o0;
            o0 = cz;
          }
          if constexpr (U & 1) {  // an odd chunk: the next one starts on the other parity
            pa ^= 1;
            pb ^= 1;
            oxa ^= oxx;
            oxb ^= oxx;
          }
        }
      }
      return;
    }
  }
  const int cnt = geo.count(c);
  for (int hh = tid; hh < cnt; hh += tp) {
    int nb[Geom::NNB];
    int nn;
    const int i = geo.site(hh, c, nb, nn);
    attempt<Real, Geom::NNB, kMeas, kEnergy>(static_cast<uint32_t>(i), pre, key, own, oth,
                                             hh, nb, nn, cp, accepted, part);
  }
}

// The sums that a measurement half-sweep of tm threads adds up, from the spins
// after the sweep, in the same order: colour 0's magnetisation, or (kBonds)
// colour 1's and, with its local fields, the bond energy.  Bound by latency (only
// tm threads have work): a unit's table entry is fetched one unit ahead and a
// chunk's spins before its first addition.
template <class Geom, bool kBonds>
__device__ __forceinline__ void sum_sites(const Geom& geo, const float* sp, int tid, int tm, int K, const int4* units,
                                          Partials<float>& part) {
  constexpr int HP = Geom::HP, LL = 2 * Geom::HL, NH = HP * LL;
  // planes taken together: a whole chunk, or a part of it (U = 8 and 6: half)
  constexpr int kChunk = kColumnChunk<float, Geom>, U = kChunk % 4 == 0 ? 4 : kChunk % 3 == 0 ? 3 : kChunk;
  constexpr int c = kBonds ? 1 : 0;
  const int S = geo.stride(), seg = LL / K;
  const SpinView<float> own(const_cast<float*>(sp) + c * 3 * S, S), oth(const_cast<float*>(sp) + (1 - c) * 3 * S, S);
  // each unit's table entry is fetched while the one before is added up
  auto entry = [&](int u) { return units != nullptr ? __ldg(units + u) : column_unit(LL, K, u); };
  int4 next = tid < HP * K ? entry(tid) : int4{};
#pragma unroll 1
  for (int u = tid; u < HP * K; u += tm) {
    const int4 d = next;
    if (u + tm < HP * K) next = entry(u + tm);
    int hh = d.x & 0x7fffffff;
    int oxa = d.y >> 24, oxb = (d.y << 8) >> 24;  // colour 1's
    V3<float> o0{}, mz{};
    if constexpr (kBonds) {
      o0 = oth.ld(hh);
      mz = oth.ld(d.y & 0xffff);
    }
#pragma unroll 1
    for (int zc = 0; zc < seg; zc += U) {
      V3<float> n[U], f[U];
#pragma unroll
      for (int k = 0; k < U; ++k, hh += HP) {
        n[k] = own.ld(hh);
        if constexpr (kBonds) {
          const int nxo = hh + ((k & 1) ? oxb : oxa);
          const int zn = (k == U - 1 && hh + HP >= NH) ? hh + HP - NH : hh + HP;
          const V3<float> cz = oth.ld(zn);
          f[k] = add3(add3(add3(add3(add3(o0, oth.ld(nxo)), oth.ld(hh + d.z)), oth.ld(hh + d.w)), cz), mz);
          mz = o0;
          o0 = cz;
        }
      }
#pragma unroll
      for (int k = 0; k < U; ++k) {
        part.mx += n[k].x;
        part.my += n[k].y;
        part.mz += n[k].z;
        if constexpr (kBonds) part.eb += Arith<float>::dot(n[k].x, n[k].y, n[k].z, f[k].x, f[k].y, f[k].z);
      }
      if constexpr (U & 1) {
        const int t = oxa;
        oxa = oxb;
        oxb = t;
      }
    }
  }
}

// ----------------------------------------------------------- measurement --
// Per-path measurement state in the path's shared-memory slice: the FP64
// accumulators and the partial-sum ring.  ring[half][slot][warp][4] holds each
// warp's partial sums (E_bond, Mx, My, Mz) of one measurement sweep; a half of
// R sweeps is flushed into the FP64 accumulators by all warps together after
// the next barrier while the other half fills, so no warp carries the
// bookkeeping alone and no FP64 operation runs per sweep.
// kFix (FP64 simple cubic lattices in shared memory): the partial sums are
// 96-bit integers, added up exactly over the warps and rounded once, so that a
// path's record does not depend on how many threads ran it: the planner chooses
// them by the paths per SM, and processes that each run a part of an ensemble
// reproduce one that runs all.  Elsewhere the number depends on the lattice alone.
template <typename Real, bool kFix = false>
struct Meter {
  double* acc;
  Real* red;
  int R, nwarps, lane, warp, tid;
  double invN;
  Real J, hf;
  int64_t j_first;  // first measurement sweep of this call (earlier ones are already flushed)
  // ring slot of the next measurement sweep j to record, ((j / R) & 1) * R +
  // j % R, kept in a 32-bit counter that advances one sweep at a time (no
  // 64-bit division per sweep); start() sets it for j_first
  int cur = 0;
  // partial sums per sweep (one per warp of the path: nwarps, or twice that
  // when two CTAs of a cluster hold the lattice), and the first of them this
  // CTA's warps write (the partner CTA writes into the owner's ring)
  int nslot = 0, slot_off = 0;
  bool pair_form = false;  // |m|^2 rounded as the two-CTA form's records have it

  __device__ void start() {
    if (nslot == 0) nslot = nwarps;
    cur = static_cast<int>(((j_first / R) & 1) * R + j_first % R);
  }
  // first of the kRedSlots partial sums of ring slot q
  __device__ Real* at(int q) const { return red + (q * nslot) * kRedSlots; }
  __device__ int slot(int64_t j) const { return static_cast<int>(((j / R) & 1) * R + (j % R)); }
  __device__ Real* cur_slot() const { return at(cur); }
  // the same of warp w, as words (kFix)
  __device__ uint32_t* words(int q, int w) const {
    return reinterpret_cast<uint32_t*>(red) + (q * nslot + w) * (kRedBytesFix / 4);
  }
  __device__ void advance() {
    if (++cur == 2 * R) cur = 0;
  }
  // Per-site observables (Sec. 2.2) of one measurement sweep from its slot.
  __device__ void observe(int q, Real& e, Real& ex, Real& ey, Real& ez) const {
    Real E = Real(0), MX = Real(0), MY = Real(0), MZ = Real(0);
    if constexpr (kFix) {
      Wide wE, wX, wY, wZ;
      for (int w = 0; w < nslot; ++w) {
        const uint4* p = reinterpret_cast<const uint4*>(words(q, w));
        const uint4 a = p[0], b = p[1], c = p[2];
        wE.add(a.x, a.y, a.z);
        wX.add(a.w, b.x, b.y);
        wY.add(b.z, b.w, c.x);
        wZ.add(c.y, c.z, c.w);
      }
      E = wE.real(kEnergyBits);
      MX = wX.real(kFixBits);
      MY = wY.real(kFixBits);
      MZ = wZ.real(kFixBits);
    } else {
      const Real* sl = at(q);
      for (int w = 0; w < nslot; ++w) {
        E += sl[w * kRedSlots + 0];
        MX += sl[w * kRedSlots + 1];
        MY += sl[w * kRedSlots + 2];
        MZ += sl[w * kRedSlots + 3];
      }
    }
    const Real rN = static_cast<Real>(invN);
    // (FP64: roundings spelled out, for the same record from either flush)
    if constexpr (sizeof(Real) == 8) e = __dmul_rn(__fma_rn(-J, E, __dmul_rn(-hf, MZ)), rN);
    else e = (-J * E - hf * MZ) * rN;
    ex = MX * rN;
    ey = MY * rN;
    ez = MZ * rN;
  }
  // Store this warp's partials of the current measurement sweep and move to
  // the next (every lane calls, once per measurement sweep, in order).
  // FP64 form: the warp's sums are exact integers; lane k < 4 has sum k.
  __device__ void record(Partials<double> part) {
    // lanes 0 .. 3: E, M_y, M_x, M_z
    const Wide v = warp_sums(part.eb, part.mx, part.my, part.mz, lane);
    if (lane < 4) {
      const int k = lane == 1 ? 2 : lane == 2 ? 1 : lane;
      if constexpr (kFix) {
        uint32_t* r = words(cur, slot_off + warp) + 3 * k;
        r[0] = v.w0;
        r[1] = v.w1;
        r[2] = v.w2;
      } else {
        (cur_slot() + (slot_off + warp) * kRedSlots)[k] = v.real(lane == 0 ? kEnergyBits : kFixBits);
      }
    }
    advance();
  }
  __device__ void record(Partials<float> part) {
    using A = Arith<float>;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      part.eb += A::shfl(part.eb, o);
      part.mx += A::shfl(part.mx, o);
      part.my += A::shfl(part.my, o);
      part.mz += A::shfl(part.mz, o);
    }
    if (lane == 0) {
      Real* r = cur_slot() + (slot_off + warp) * kRedSlots;
      r[0] = part.eb;
      r[1] = part.mx;
      r[2] = part.my;
      r[3] = part.mz;
    }
    advance();
  }
  // a b, rounded by itself in FP64 (whatever is added to it later).
  static __device__ __forceinline__ Real product(Real a, Real b) {
    if constexpr (sizeof(Real) == 8) return __dmul_rn(a, b);
    else return a * b;
  }
  // The same by one warp in a third of the FP64 instructions (76 cycles each,
  // and a small lattice's flush is a good part of its sweeps): lanes l and
  // l + 16 take sweep j0 + l, each half of the observables, and the 16 sweeps
  // are summed by exchanges that halve what a lane carries, in flush's order.
  __device__ void flush_warp(int64_t j0, int n) const {
    Real e = Real(0), ex = Real(0), ey = Real(0), ez = Real(0);
    const int l = lane & 15;
    const bool upper = lane >= 16;
    if (l < n) observe(slot(j0 + l), e, ex, ey, ez);
    const Real m2 = Arith<Real>::square(ex, ey, ez), m = sqrt(m2);
    // lower half: E E2 M M2 M4 MX MY; upper half: MZ MZ2 |MZ| EM EMZ MMZ
    Real v[8];
    const Real p = upper ? ez : e;
    v[0] = p;
    v[1] = product(p, p);
    v[2] = upper ? fabs(ez) : m;
    v[3] = upper ? product(e, m) : m2;
    v[4] = upper ? product(e, ez) : product(m2, m2);
    v[5] = upper ? product(m, ez) : ex;
    v[6] = upper ? Real(0) : ey;
    v[7] = Real(0);
#pragma unroll
    for (int w = 4; w >= 1; w >>= 1) {  // lane bit w: keep the upper w values, give away the lower
      const bool up = lane & w;
#pragma unroll
      for (int k = 0; k < w; ++k) {
        const Real give = up ? v[k] : v[k + w], keep = up ? v[k + w] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, give, w);
      }
    }
    const Real total = v[0] + __shfl_xor_sync(0xffffffffu, v[0], 8);  // value (lane & 7) of this half
    const int at = (lane & 7) + (upper ? static_cast<int>(MP_R_MZ) : static_cast<int>(MP_R_E));
    static_assert(MP_R_MY == 6 && MP_R_MZ == 7 && MP_R_MMZ == 12, "record order");
    if (!(lane & 8) && (lane & 7) < (upper ? 6 : 7)) acc[at] += total;
  }
  // Flush sweeps j0 .. j0+n-1 (one ring half): lane l takes sweep j0+l; warp
  // w owns observables w, w + warps, ...; each owned observable is summed
  // over the lanes and added to its FP64 accumulator.
  // FP64 form with one warp and a ring of 16: flush_warp.
  __device__ void flush(int64_t j0, int n) const {
    using A = Arith<Real>;
    if constexpr (sizeof(Real) == 8) {
      if (nwarps == 1 && nslot == 1 && R == 16) {
        flush_warp(j0, n);
        return;
      }
    }
    Real e = Real(0), ex = Real(0), ey = Real(0), ez = Real(0);
    if (lane < n) observe(slot(j0 + lane), e, ex, ey, ez);
    Real m2;
    if constexpr (sizeof(Real) == 4) m2 = pair_form ? A::square_pair(ex, ey, ez) : A::square(ex, ey, ez);
    else m2 = A::square(ex, ey, ez);
    const Real m = sqrt(m2);
    for (int k = warp; k <= MP_R_MMZ; k += nwarps) {
      Real v;
      switch (k) {  // k is the same in every lane of the warp
        case MP_R_E: v = e; break;
        case MP_R_E2: v = product(e, e); break;
        case MP_R_M: v = m; break;
        case MP_R_M2: v = m2; break;
        case MP_R_M4: v = product(m2, m2); break;
        case MP_R_MX: v = ex; break;
        case MP_R_MY: v = ey; break;
        case MP_R_MZ: v = ez; break;
        case MP_R_MZ2: v = product(ez, ez); break;
        case MP_R_AMZ: v = fabs(ez); break;
        case MP_R_EM: v = product(e, m); break;
        case MP_R_EMZ: v = product(e, ez); break;
        default: v = product(m, ez); break;  // MP_R_MMZ
      }
      if (lane >= n) v = Real(0);
      // FP64: in flush_warp's order (a path of one warp may take either)
      constexpr int kOrder[2][5] = {{16, 8, 4, 2, 1}, {16, 4, 2, 1, 8}};
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const int o = kOrder[sizeof(Real) == 8][q];
        if (o < R) v += A::shfl(v, o);
      }
      if (lane == 0) acc[k] += static_cast<double>(v);
    }
  }
  static __device__ __noinline__ void flush_call(Meter m, int64_t j0, int n) { m.flush(j0, n); }
  // At measurement sweep j (the current one), after its first barrier: flush
  // the previous half.  kCall: as a call, which leaves the sweep loop the
  // registers that the integer sums would take: FP64 L = 16, 3072 paths, 200 sweeps:
  // 39.1 -> 38.5 ms, L = 12 and 20 1.7% (not the one-site form: 1.21 -> 1.26 ms).
  template <bool kCall = false>
  __device__ void maybe_flush(int64_t j) const {
    if ((cur == 0 || cur == R) && j > j_first) {
      const int64_t j0 = j - R > j_first ? j - R : j_first;
      if constexpr (kCall) flush_call(*this, j0, static_cast<int>(j - j0));
      else flush(j0, static_cast<int>(j - j0));
    }
  }
  // After the call's last sweep and its barrier: flush the rest of the
  // measurement sweeps j_first .. n_meas-1 and keep the final state.
  __device__ void finish(int64_t n_meas) const {
    const int64_t last = n_meas - 1;
    if (last < j_first) return;  // no measurement sweep in this call
    int64_t j0 = last - last % R;
    if (j0 < j_first) j0 = j_first;
    flush(j0, static_cast<int>(last - j0) + 1);
    if (tid == 0) {  // the final state: the paper's per-path output
      Real e, ex, ey, ez;
      observe(slot(last), e, ex, ey, ez);
      acc[MP_R_FMX] = static_cast<double>(ex);
      acc[MP_R_FMY] = static_cast<double>(ey);
      acc[MP_R_FMZ] = static_cast<double>(ez);
      acc[MP_R_FE] = static_cast<double>(e);
    }
  }
  // Reduce the acceptance count and the worst | |S| - 1 | over the group's warps
  // (nwarps, or all_warps of a wide path) and
  // write the path's record (the ring area is reused; call after a barrier).
  __device__ void write_record(double* rec, int accepted, double worst, int64_t nsweeps,
                               int64_t n_meas, int N, int tp, int bar, double accepted_before,
                               double* save_accepted, int all_warps = 0) const {
    double nacc = static_cast<double>(accepted);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      nacc += __shfl_xor_sync(0xffffffffu, nacc, o);
      worst = fmax(worst, __shfl_xor_sync(0xffffffffu, worst, o));
    }
    double* fin = reinterpret_cast<double*>(red);  // 2 doubles per warp
    if (lane == 0) {
      fin[2 * warp + 0] = nacc;
      fin[2 * warp + 1] = worst;
    }
    group_sync(tp, bar);
    if (tid == 0) {
      double tot = accepted_before, wmax = 0.0;
      for (int w = 0; w < (all_warps > 0 ? all_warps : nwarps); ++w) {
        tot += fin[2 * w + 0];
        wmax = fmax(wmax, fin[2 * w + 1]);
      }
      if (save_accepted) *save_accepted = tot;
      const double inv = n_meas > 0 ? 1.0 / static_cast<double>(n_meas) : NAN;
      for (int k = MP_R_E; k <= MP_R_MMZ; ++k) rec[k] = acc[k] * inv;
      for (int k = MP_R_FMX; k <= MP_R_FE; ++k) rec[k] = acc[k];
      rec[MP_R_ACC] = tot / (static_cast<double>(nsweeps) * static_cast<double>(N));
      rec[MP_R_NORM] = wmax;
      rec[MP_R_SPARE] = 0.0;
    }
  }
};

// The measurement state of a path in a geometry: exact sums where the number of
// threads may go by the load; those sweeps also call the flush.
template <typename Real, class Geom>
constexpr bool kExactSums = sizeof(Real) == 8 && Geom::kColumns;

// Initial spin of site i: uniform on the sphere (Sec. 2.2), uniform angles,
// or the ordered start of Sec. 5.
template <typename Real>
__device__ __forceinline__ V3<Real> initial_spin(uint32_t i, uint32_t c2, uint32_t c3i, const SweepParams& P,
                                                 int mode) {
  using S = Stored<Real>;
  const Philox4 r = philox4x32_10(i, 0u, c2, c3i, P.key);
  if (mode == MP_INIT_ORDERED) return V3<Real>{S::from(Real(0)), S::from(Real(0)), S::from(Real(1))};
  Real x, y, z;
  if (mode == MP_INIT_ANGLES) {
    Arith<Real>::init_angles(r.x, r.y, x, y, z);
  } else if constexpr (sizeof(Real) == 8) {
    const Fix3 t = fix_trial(r.x, r.y, fix_root(r.x), sine_shared());
    return V3<Real>{t.x, t.y, t.z};
  } else {
    Arith<Real>::trial(r.x, r.y, x, y, z);
  }
  return V3<Real>{S::from(x), S::from(y), S::from(z)};
}

// --------------------------------------------------------- resumable state --
// A path's state in HBM (resumable runs): [acc: 24 doubles][accepted: double]
// padded to kStateHeader bytes, then its spins.
__device__ __forceinline__ unsigned char* path_state(const SweepParams& P, int sys_idx, int64_t path) {
  return P.state ? P.state + P.state_offset[sys_idx] + path * P.state_stride[sys_idx] : nullptr;
}

// Poll of the host's cancel flag by one thread of the group, every kCancelPoll
// sweeps of a call; the group reads the verdict after its next barrier.
__device__ __forceinline__ void poll_cancel(const SweepParams& P, int64_t s, int tid, int* flag) {
  if (tid == 0 && P.cancel != nullptr && ((s - P.s_begin) % kCancelPoll) == 0 && *P.cancel != 0) {
    *flag = 1;
    atomicExch(P.error, kErrCanceled);
  }
}

// Each thread group's cancel verdict; one array for all paths of a geometry
// (a second one would take shared memory, and rings of partial sums, from them).
template <typename Real, class Geom>
__device__ __forceinline__ int* cancel_flags() {
  __shared__ int flags[kMaxGroups];
  return flags;
}

// ------------------------------------------------------------- one path --
// The lattice lives in the slice's shared memory, or in HBM at `hbm_spins`
// (the same layout) when it is updated in place there.
//
// kOne: every thread owns at most one site of each colour (tp >= sites per
// colour: short chains, L <= 4).  A sweep then waits on the latency of two
// attempts, most of it in their random numbers and trial spins, which do not
// depend on the lattice: both colours' are drawn together, before the first
// update, and neighbours are decoded once per path.
// FP64 L = 4, 256 paths: 1.31 -> 0.98 us per sweep; FP32 with 2000 paths 9.9e10 -> 1.3e11
// attempts/s.
//
// FP32 sums depend on their order, which is that of tm threads each taking its
// sites in turn.  Where a launch has too few paths, or paths too large, for
// that many threads to fill the SM (the planner's wide_threads), the path gets
// tp > tm threads: all of them update, and in a measurement sweep the first tm
// then add up the sums from the new spins (sum_sites).  One path per SM, half of
// the sweeps measured: L = 10 2.5e10 -> 5.1e10 attempts/s (32 threads, now 256), L =
// 20 1.1e11 -> 1.7e11 (160, now 512); with thermalisation alone 2.6e10 -> 9.4e10 and
// 1.15e11 -> 2.14e11.
// kWide paths have a body of their own: with a branch in the common one, measured
// sweeps of the others lost 2%.
template <typename Real, class Geom, bool kOne = false, bool kWide = false>
__device__ __forceinline__ void run_path(const Geom geo, const DevSystem& sy, int sys_idx,
                                         int64_t path, const SweepParams& P, unsigned char* slice,
                                         int tid, int tp, int bar, Real* hbm_spins = nullptr) {
  static_assert(!kWide || (sizeof(Real) == 4 && Geom::kColumns && !kOne), "wide paths are FP32 column walks");
  constexpr bool kExact = kExactSums<Real, Geom>;
  Real* sp = hbm_spins;
  if (!sp) sp = reinterpret_cast<Real*>(slice + slice_spin_offset(tp, sy.ring, kExact ? kRedBytesFix : kRedBytes));
  const int S = geo.stride();
  const uint32_t c2 = static_cast<uint32_t>(sy.path_begin + path);  // path id
  const uint32_t c3u = kTagUpdate | (static_cast<uint32_t>(sys_idx) << 8);
  const uint32_t c3i = kTagInit | (static_cast<uint32_t>(sys_idx) << 8);
  const int init = path_init_mode(P.init_mode, path, sy.n_paths);
  const Real J = static_cast<Real>(sy.J), hf = static_cast<Real>(sy.h);
  const Couplings<Real> cp(P.systems + sys_idx);
  // column segments per column (column_segments; 0 = decode every site: open
  // chains), and the host's table of the column-walk units when it was made
  // for this chunk (the table's K is then that of the same rule)
  int K = 0;
  const int4* units = nullptr;
  if constexpr (Geom::kColumns) {
    constexpr int LL = 2 * Geom::HL;
    constexpr int U = kColumnChunk<Real, Geom>;
    static_assert(LL % U == 0, "a whole column is a whole number of chunks");
    static_assert(Geom::HP * LL < 65536, "unit tables hold half indices in 16 bits");
    if (P.units != nullptr && sy.unit_off >= 0 && sy.unit_U == U && sy.unit_K > 0) {
      K = sy.unit_K;
      units = P.units + sy.unit_off;
    } else {
      K = column_segments(LL, U, tp);
    }
  }
  const int64_t j_first = P.s_begin > P.n_therm ? P.s_begin - P.n_therm : 0;
  Meter<Real, kExact> meter{reinterpret_cast<double*>(slice + slice_acc_offset()),
                    reinterpret_cast<Real*>(slice + slice_red_offset()),
                    sy.ring, (kWide ? sy.tm : tp) >> 5, tid & 31, tid >> 5, tid,
                    1.0 / static_cast<double>(sy.N), J, hf, j_first};
  meter.start();
  unsigned char* st = path_state(P, sys_idx, path);
  Real* st_spins = st ? reinterpret_cast<Real*>(st + kStateHeader) : nullptr;
  typename Stored<Real>::C* raw = reinterpret_cast<typename Stored<Real>::C*>(sp);
  int* const cancel_flag = cancel_flags<Real, Geom>();
  const int gidx = bar - 1;

  if (P.resume && st) {  // continue from the saved state
    for (int k = tid; k < 6 * S; k += tp) raw[k] = Stored<Real>::from(st_spins[k]);
    if (tid < kAccDoubles) meter.acc[tid] = reinterpret_cast<const double*>(st)[tid];
  } else {
    for (int c = 0; c < 2; ++c) {
      const SpinView<Real> own(sp + c * 3 * S, S);
      const int cnt = geo.count(c);
      for (int hh = tid; hh < cnt; hh += tp) {
        int nb[Geom::NNB];
        int nn;
        const int i = geo.site(hh, c, nb, nn);
        const V3<Real> v = initial_spin<Real>(static_cast<uint32_t>(i), c2, c3i, P, init);
        own.st(hh, v.x, v.y, v.z);
      }
    }
    if (tid < kAccDoubles) meter.acc[tid] = 0.0;
  }
  const double accepted_before =
      (P.resume && st) ? reinterpret_cast<const double*>(st)[kAccDoubles] : 0.0;
  if (tid == 0) cancel_flag[gidx] = 0;
  group_sync(tp, bar);

  int accepted = 0;
  bool canceled = false;
  if constexpr (kOne) {
    const SpinView<Real> view[2] = {SpinView<Real>(sp, S), SpinView<Real>(sp + 3 * S, S)};
    bool act[2];
    int h[2], nb[2][Geom::NNB], nn[2];
    uint32_t site[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      act[c] = tid < geo.count(c);
      h[c] = act[c] ? tid : 0;
      site[c] = static_cast<uint32_t>(geo.site(h[c], c, nb[c], nn[c]));
    }
    auto field = [&](auto c_c) {
      constexpr int c = decltype(c_c)::value;
      V3<Real> f{};
#pragma unroll
      for (int j = 0; j < Geom::NNB; ++j)
        if (j < nn[c]) f = add3(f, view[1 - c].ld(nb[c][j]));
      return f;
    };
    constexpr std::integral_constant<int, 0> c_0{};
    constexpr std::integral_constant<int, 1> c_1{};
    for (int64_t s = P.s_begin; s < P.s_end; ++s) {
      const PhiloxPrefix pre = philox_prefix(static_cast<uint32_t>(s), c2, c3u, P.key);
      const Ahead<Real> d0(philox4x32_10(site[0], pre, P.key)), d1(philox4x32_10(site[1], pre, P.key));
      Partials<Real> part;
      poll_cancel(P, s, tid, &cancel_flag[gidx]);
      const bool meas = s >= P.n_therm;
      if (meas) d0.template apply<true, false>(view[0], h[0], field(c_0), cp, act[0], accepted, part);
      else d0.template apply<false, false>(view[0], h[0], field(c_0), cp, act[0], accepted, part);
      group_sync(tp, bar);
      if (cancel_flag[gidx]) {
        canceled = true;
        break;
      }
      if (meas) {
        meter.maybe_flush(s - P.n_therm);
        d1.template apply<true, true>(view[1], h[1], field(c_1), cp, act[1], accepted, part);
        meter.record(part);
      } else {
        d1.template apply<false, false>(view[1], h[1], field(c_1), cp, act[1], accepted, part);
      }
      group_sync(tp, bar);
    }
  } else
  for (int64_t s = P.s_begin; s < P.s_end; ++s) {
    const uint32_t sw = static_cast<uint32_t>(s);
    const PhiloxPrefix pre = philox_prefix(sw, c2, c3u, P.key);
    Partials<Real> part;
    poll_cancel(P, s, tid, &cancel_flag[gidx]);
    if (kWide || s < P.n_therm) {
      half_sweep<Real, Geom, false, false>(geo, 0, pre, P.key, sp, tid, tp, K, units, cp, accepted, part);
      group_sync(tp, bar);
      if (cancel_flag[gidx]) {
        canceled = true;
        break;
      }
      half_sweep<Real, Geom, false, false>(geo, 1, pre, P.key, sp, tid, tp, K, units, cp, accepted, part);
      group_sync(tp, bar);
      if constexpr (kWide) {
        if (s >= P.n_therm) {
          if (tid < sy.tm) {  // whole warps
            meter.maybe_flush(s - P.n_therm);
            const bool table = units != nullptr;
            const int sum_K = table ? sy.sum_K : column_segments(2 * Geom::HL, kColumnChunk<Real, Geom>, sy.tm);
            const int4* sum_units = table ? P.units + sy.sum_off : nullptr;
            sum_sites<Geom, false>(geo, sp, tid, sy.tm, sum_K, sum_units, part);
            sum_sites<Geom, true>(geo, sp, tid, sy.tm, sum_K, sum_units, part);
            meter.record(part);
          }
          group_sync(tp, bar);
        }
      }
      continue;
    }
    if constexpr (!kWide) {
      // Measurement sweep j.  Colour-0 sites keep their values during the
      // colour-1 pass, so the colour-1 local fields give every bond once.
      const int64_t j = s - P.n_therm;
      half_sweep<Real, Geom, true, false>(geo, 0, pre, P.key, sp, tid, tp, K, units, cp, accepted, part);
      group_sync(tp, bar);
      if (cancel_flag[gidx]) {
        canceled = true;
        break;
      }
      meter.template maybe_flush<kExact>(j);
      half_sweep<Real, Geom, true, true>(geo, 1, pre, P.key, sp, tid, tp, K, units, cp, accepted, part);
      meter.record(part);
      group_sync(tp, bar);
    }
  }
  if (canceled) {  // the call is discarded: no record, no saved state
    group_sync(tp, bar);
    return;
  }
  const int64_t n_meas_done = P.s_end > P.n_therm ? P.s_end - P.n_therm : 0;
  if (!kWide || (tid >> 5) < meter.nwarps) meter.finish(n_meas_done);
  group_sync(tp, bar);

  Real worst = Real(0);
  for (int c = 0; c < 2; ++c) {
    const SpinView<Real> own(sp + c * 3 * S, S);
    for (int hh = tid; hh < geo.count(c); hh += tp) {
      const V3<Real> v = own.ld(hh);
      worst = fmax(worst, norm_error(v));
    }
  }
  if (P.save && st) {
    for (int k = tid; k < 6 * S; k += tp) st_spins[k] = Stored<Real>::real(raw[k]);
    if (tid < kAccDoubles) reinterpret_cast<double*>(st)[tid] = meter.acc[tid];
  }
  meter.write_record(P.records + (sy.rec_offset + path) * MP_NREC, accepted,
                     static_cast<double>(worst), P.s_end, n_meas_done, sy.N, tp, bar,
                     accepted_before, (P.save && st) ? reinterpret_cast<double*>(st) + kAccDoubles : nullptr,
                     kWide ? tp >> 5 : 0);
  if (P.spins != nullptr) {
    double* out = P.spins + P.spin_offset[sys_idx] + path * 3 * static_cast<int64_t>(sy.N);
    for (int c = 0; c < 2; ++c) {
      const SpinView<Real> own(sp + c * 3 * S, S);
      for (int hh = tid; hh < geo.count(c); hh += tp) {
        int nb[Geom::NNB];
        int nn;
        const int i = geo.site(hh, c, nb, nn);
        const V3<Real> v = own.ld(hh);
        out[3 * i + 0] = Stored<Real>::real(v.x);
        out[3 * i + 1] = Stored<Real>::real(v.y);
        out[3 * i + 2] = Stored<Real>::real(v.z);
      }
    }
  }
  group_sync(tp, bar);  // the slice is reused by the next item
}

// ------------------------------------------------ two-CTA clusters -------
// A simple cubic lattice too large for one SM's shared memory but not for
// two (FP32 L = 32: 393 KB of spins) is held by the two CTAs of a cluster:
// CTA rank r keeps the z-planes r L/2 .. r L/2 + L/2 - 1, and in each colour
// array also one halo plane on either side (local planes 0 and L/2 + 1) with
// the partner's boundary plane.  A half-sweep of colour c updates the local
// planes by the same column walk as run_path (the halo planes give the +-z
// neighbours across the cut, so no index wraps in z), and each thread pushes
// the new values of its column's two boundary sites straight into the
// partner's halo planes of colour c (distributed shared memory stores).  The
// partner reads colour c only in the next half-sweep, after the cluster
// barrier that ends this one, so one barrier per half-sweep orders
// everything; during a half-sweep each CTA reads only colour 1 - c and writes
// only colour c.  Measurement partials of the partner's warps go into the
// owner's (rank 0's) partial-sum ring, which then holds every warp of the
// lattice; rank 0 flushes, keeps the FP64 accumulators and writes the record.
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t n;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
  return n;
}
// Generic address of the same shared-memory location in CTA `rank` of the cluster.
template <typename T>
__device__ __forceinline__ T* map_rank(T* p, uint32_t rank) {
  uint64_t out;
  asm volatile("mapa.u64 %0, %1, %2;" : "=l"(out) : "l"(reinterpret_cast<uint64_t>(p)), "r"(rank));
  return reinterpret_cast<T*>(out);
}
// Every thread of both CTAs; release/acquire at cluster scope, so shared
// memory written (locally or remotely) before it is visible after it.
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

template <int L>
struct PairGeom {
  static constexpr int HL = L / 2, HP = L * L / 2;
  static constexpr int ZL = L / 2;       // planes per CTA
  static constexpr int S = HP * (ZL + 2);  // sites per colour array, with the two halo planes
  static_assert(6 * S * 4 == pair_spin_bytes(L, 4), "pair layout");
};

// Planes of a column walked per unrolled chunk (even, so that each site's x
// parity is fixed at compile time): 8, 0.4% faster than 4 on the batch of
// uneven sizes.
constexpr int kPairChunk = 8;

template <typename Real, int L, bool kMeas, bool kEnergy>
__device__ __forceinline__ void half_sweep_pair(int c, int zbase, const PhiloxPrefix& pre,
                                                const PhiloxKeys& key, Real* sp, Real* partner_sp,
                                                int tid, int tp, const Couplings<Real>& cp,
                                                int& accepted, Partials<Real>& part) {
  using G = PairGeom<L>;
  constexpr int HL = G::HL, HP = G::HP, ZL = G::ZL, S = G::S;
  const SpinView<Real> own(sp + c * 3 * S, S), oth(sp + (1 - c) * 3 * S, S);
  const SpinView<Real> halo(partner_sp + c * 3 * S, S);  // the partner's array of colour c
  for (int col = tid; col < HP; col += tp) {
    const int hx = col % HL;
    const int y = col / HL;
    const int oyp = (y == L - 1) ? -(L - 1) * HL : HL;
    const int oym = (y == 0) ? (L - 1) * HL : -HL;
    const int oxp1 = (hx == HL - 1) ? -(HL - 1) : 1;  // +x offset when x is odd
    const int oxm0 = (hx == 0) ? (HL - 1) : -1;         // -x offset when x is even
    // x parity of the sites in local planes 1, 3, ... (pa) and 2, 4, ... (pb):
    // chunks have an even number of planes, so within one the choice of
    // parity and x-neighbour offset is made at compile time
    const int pa = (y + zbase + c) & 1, pb = pa ^ 1;
    const int oxa = pa ? oxp1 : oxm0, oxb = pa ? oxm0 : oxp1;
    int hh = col + HP;                                   // local plane 1
    V3<Real> o0 = oth.ld(hh);       // the other colour at the site's half index
    V3<Real> mz = oth.ld(hh - HP);  // -z neighbour (halo plane 0)
    static_assert(kPairChunk % 2 == 0 && ZL % kPairChunk == 0, "even chunks that tile the planes");
    for (int zc = 0; zc < ZL; zc += kPairChunk) {
#pragma unroll
      for (int k = 0; k < kPairChunk; ++k, hh += HP) {
        // global plane zbase + zc + k
        const int p = (k & 1) ? pb : pa;
        const int nxo = hh + ((k & 1) ? oxb : oxa);
        const V3<Real> cz = oth.ld(hh + HP);
        const V3<Real> f =
            add3(add3(add3(add3(add3(o0, oth.ld(nxo)), oth.ld(hh + oyp)), oth.ld(hh + oym)), cz), mz);
        // site index x + L(y + L z_global) = 2 (col + HP z_global) + p
        update<kMeas, kEnergy>(static_cast<uint32_t>(2 * (hh + HP * (zbase - 1)) + p), pre, key, own, hh, f, cp,
                               accepted, part);
        mz = o0;
        o0 = cz;
      }
    }
    // the column's boundary sites to the partner's halo planes: local plane 1
    // is the partner's plane ZL + 1, local plane ZL its plane 0
    const V3<Real> a = own.ld(col + HP);
    halo.st(col + HP * (ZL + 1), a.x, a.y, a.z);
    const V3<Real> b = own.ld(col + HP * ZL);
    halo.st(col, b.x, b.y, b.z);
  }
}

// One path of a simple cubic L (= kPairL) lattice on the two CTAs of a
// cluster; every thread of both CTAs calls it with the same arguments except
// `rank` and tid.  The record, the saved accumulators and the acceptance
// count are written by rank 0; each rank saves and outputs its own planes.
template <typename Real, int L>
__device__ void run_path_pair(const DevSystem& sy, int sys_idx, int64_t path, const SweepParams& P,
                              unsigned char* slice, int tid, int tp, uint32_t rank) {
  using G = PairGeom<L>;
  constexpr int HL = G::HL, HP = G::HP, ZL = G::ZL, S = G::S;
  constexpr int NH = L * L * L / 2;  // sites per colour of the whole lattice
  // rank 0's ring holds the partials of both CTAs' warps
  Real* sp = reinterpret_cast<Real*>(slice + slice_spin_offset(2 * tp, sy.ring, kRedBytes));
  Real* partner_sp = map_rank(sp, rank ^ 1u);
  const int zbase = static_cast<int>(rank) * ZL;
  const uint32_t c2 = static_cast<uint32_t>(sy.path_begin + path);  // path id
  const uint32_t c3u = kTagUpdate | (static_cast<uint32_t>(sys_idx) << 8);
  const uint32_t c3i = kTagInit | (static_cast<uint32_t>(sys_idx) << 8);
  const int init = path_init_mode(P.init_mode, path, sy.n_paths);
  const Real J = static_cast<Real>(sy.J), hf = static_cast<Real>(sy.h);
  const Couplings<Real> cp(P.systems + sys_idx);
  const int64_t j_first = P.s_begin > P.n_therm ? P.s_begin - P.n_therm : 0;
  Real* red0 = reinterpret_cast<Real*>(slice + slice_red_offset());
  Meter<Real> meter{reinterpret_cast<double*>(slice + slice_acc_offset()),
                    rank == 0 ? red0 : map_rank(red0, 0u),
                    sy.ring, tp >> 5, tid & 31, tid >> 5, tid,
                    1.0 / static_cast<double>(sy.N), J, hf, j_first};
  meter.nslot = 2 * (tp >> 5);
  meter.pair_form = true;
  meter.slot_off = rank == 0 ? 0 : (tp >> 5);
  meter.start();
  unsigned char* st = path_state(P, sys_idx, path);
  Real* st_spins = st ? reinterpret_cast<Real*>(st + kStateHeader) : nullptr;
  __shared__ int pair_cancel;
  __shared__ double pair_xch[2];  // rank 1's acceptance count and worst | |S| - 1 |, on rank 0
  const bool resume = P.resume && st;

  // local plane zl holds global plane (zbase + zl - 1) mod L, zl = 0 .. ZL + 1
  for (int c = 0; c < 2; ++c) {
    const SpinView<Real> own(sp + c * 3 * S, S);
    for (int h = tid; h < S; h += tp) {
      const int col = h % HP, zl = h / HP;
      const int zg = (zbase + zl - 1 + L) % L;
      const int hg = col + HP * zg;  // half index in the whole lattice
      const int p = (col / HL + zg + c) & 1;
      const V3<Real> v = resume ? SpinView<Real>(st_spins + c * 3 * NH, NH).ld(hg)
                                : initial_spin<Real>(static_cast<uint32_t>(2 * hg + p), c2, c3i, P, init);
      own.st(h, v.x, v.y, v.z);
    }
  }
  if (tid < kAccDoubles) meter.acc[tid] = (resume && rank == 0) ? reinterpret_cast<const double*>(st)[tid] : 0.0;
  const double accepted_before = (resume && rank == 0) ? reinterpret_cast<const double*>(st)[kAccDoubles] : 0.0;
  if (tid == 0) pair_cancel = 0;
  cluster_sync_all();

  int accepted = 0;
  bool canceled = false;
  for (int64_t s = P.s_begin; s < P.s_end; ++s) {
    const uint32_t sw = static_cast<uint32_t>(s);
    const PhiloxPrefix pre = philox_prefix(sw, c2, c3u, P.key);
    Partials<Real> part;
    // rank 0 polls the host's flag and tells both CTAs, so that they stop together
    if (rank == 0 && tid == 0 && P.cancel != nullptr && ((s - P.s_begin) % kCancelPoll) == 0 &&
        *P.cancel != 0) {
      pair_cancel = 1;
      *map_rank(&pair_cancel, 1u) = 1;
      atomicExch(P.error, kErrCanceled);
    }
    const bool meas = s >= P.n_therm;
    if (meas)
      half_sweep_pair<Real, L, true, false>(0, zbase, pre, P.key, sp, partner_sp, tid, tp, cp, accepted, part);
    else
      half_sweep_pair<Real, L, false, false>(0, zbase, pre, P.key, sp, partner_sp, tid, tp, cp, accepted, part);
    cluster_sync_all();
    if (pair_cancel) {
      canceled = true;
      break;
    }
    if (meas) {
      if (rank == 0) meter.maybe_flush(s - P.n_therm);
      half_sweep_pair<Real, L, true, true>(1, zbase, pre, P.key, sp, partner_sp, tid, tp, cp, accepted, part);
      meter.record(part);
    } else {
      half_sweep_pair<Real, L, false, false>(1, zbase, pre, P.key, sp, partner_sp, tid, tp, cp, accepted, part);
    }
    cluster_sync_all();
  }
  if (canceled) {  // the call is discarded: no record, no saved state
    cluster_sync_all();
    return;
  }
  const int64_t n_meas_done = P.s_end > P.n_therm ? P.s_end - P.n_therm : 0;
  if (rank == 0) meter.finish(n_meas_done);
  __syncthreads();  // the ring area is free from here on (finish has read its last slot)

  // this CTA's planes: worst | |S| - 1 |, saved state, final spins
  Real worst = Real(0);
  for (int c = 0; c < 2; ++c) {
    const SpinView<Real> own(sp + c * 3 * S, S);
    for (int h = tid + HP; h < HP * (ZL + 1); h += tp) {
      const V3<Real> v = own.ld(h);
      worst = fmax(worst, norm_error(v));
      const int col = h % HP, zg = zbase + h / HP - 1;
      const int hg = col + HP * zg;
      if (P.save && st) SpinView<Real>(st_spins + c * 3 * NH, NH).st(hg, v.x, v.y, v.z);
      if (P.spins != nullptr) {
        const int i = 2 * hg + ((col / HL + zg + c) & 1);
        double* out = P.spins + P.spin_offset[sys_idx] + path * 3 * static_cast<int64_t>(sy.N) + 3 * i;
        out[0] = v.x;
        out[1] = v.y;
        out[2] = v.z;
      }
    }
  }
  // acceptance count and worst norm of this CTA; rank 1 hands its totals to rank 0
  double nacc = static_cast<double>(accepted), wst = static_cast<double>(worst);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    nacc += __shfl_xor_sync(0xffffffffu, nacc, o);
    wst = fmax(wst, __shfl_xor_sync(0xffffffffu, wst, o));
  }
  double* pair_red = reinterpret_cast<double*>(red0);  // this CTA's own ring area
  if ((tid & 31) == 0) {
    pair_red[2 * (tid >> 5)] = nacc;
    pair_red[2 * (tid >> 5) + 1] = wst;
  }
  __syncthreads();
  if (tid == 0) {
    double tot = 0.0, wmax = 0.0;
    for (int w = 0; w < (tp >> 5); ++w) {
      tot += pair_red[2 * w];
      wmax = fmax(wmax, pair_red[2 * w + 1]);
    }
    if (rank == 1) {
      double* x = map_rank(pair_xch, 0u);
      x[0] = tot;
      x[1] = wmax;
    } else {
      pair_red[0] = tot;
      pair_red[1] = wmax;
    }
  }
  cluster_sync_all();  // rank 1's totals are in rank 0's pair_xch
  if (rank == 0 && tid == 0) {
    const double tot = accepted_before + pair_red[0] + pair_xch[0];
    const double wmax = fmax(pair_red[1], pair_xch[1]);
    double* rec = P.records + (sy.rec_offset + path) * MP_NREC;
    const double inv = n_meas_done > 0 ? 1.0 / static_cast<double>(n_meas_done) : NAN;
    for (int k = MP_R_E; k <= MP_R_MMZ; ++k) rec[k] = meter.acc[k] * inv;
    for (int k = MP_R_FMX; k <= MP_R_FE; ++k) rec[k] = meter.acc[k];
    rec[MP_R_ACC] = tot / (static_cast<double>(P.s_end) * static_cast<double>(sy.N));
    rec[MP_R_NORM] = wmax;
    rec[MP_R_SPARE] = 0.0;
    if (P.save && st) {
      for (int k = 0; k < kAccDoubles; ++k) reinterpret_cast<double*>(st)[k] = meter.acc[k];
      reinterpret_cast<double*>(st)[kAccDoubles] = tot;
    }
  }
  cluster_sync_all();  // the slices (and pair_xch) are reused by the next item
}

// ------------------------------------------------------ TMA primitives --
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
// End an mbarrier's life before its memory is initialised again or reused.
__device__ __forceinline__ void mbar_inval(uint64_t* bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}
// Bulk copy global -> shared of `bytes` (multiple of 16, both addresses 16-byte
// aligned), completing on the mbarrier `bar`.
__device__ __forceinline__ void tma_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}
// Bulk copy shared -> global, as its own bulk group.
__device__ __forceinline__ void tma_store(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst),
               "r"(smem_addr(src)), "r"(bytes)
               : "memory");
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// Wait until at most N (a constant) bulk store groups may still read shared memory.
template <int N>
__device__ __forceinline__ void tma_wait_read_n() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
#define tma_wait_read(n) tma_wait_read_n<n>()
__device__ __forceinline__ void tma_wait_all() {
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}
__device__ __forceinline__ void fence_async_shared() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Wait for phase `parity` of the mbarrier, giving up after about 2 s: then the
// error flag is set and false returned (the caller stops the path cleanly).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* error) {
  const uint32_t a = smem_addr(bar);
  uint64_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    uint32_t done;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    if ((it & 63) == 0) {
      const uint64_t t = global_ns();
      if (it == 0) t0 = t;
      else if (t - t0 > 2000000000ull) {
        atomicExch(error, 1);
        return false;
      }
    }
  }
}

// ---------------------------------------------------- streamed from HBM --
// Lattices too large for shared memory.  Each path's spins stay in HBM in the
// layout [z][colour][(x, y) pairs | z][L*L/2] (a "half-plane" is one colour
// of one z-plane, padded to 16 bytes), in a buffer owned by the thread group for the
// whole run.  A sweep walks the z-planes as a wavefront over a ring of 4 + 5
// half-plane buffers in shared memory, filled by TMA bulk copies and written
// back by bulk stores:
//   step q = 0 .. L+1:  (a) colour-0 update of plane q          (q < L)
//                       (b) colour-1 update of plane (q-1) mod L (q >= 2)
// Colour 0 of plane q needs colour 1 of planes q-1, q, q+1 still old; colour 1
// of plane q-1 needs colour 0 of planes q-2, q-1, q already new; plane 0's
// colour-1 update waits until the end (it needs colour 0 of plane L-1 new,
// and colour 0 of plane L-1 needs colour 1 of plane 0 old).  Every update thus
// sees exactly the neighbour values of the two-pass checkerboard sweep.
// Phases (a) and (b) of a step run back to back, with one group barrier per
// step (see the loop below for why no barrier is needed between them).
// Ring indices: colour-0 step index q' = 0..L+1 (planes 0..L-1, 0, 1) in slot
// q' mod 4; colour-1 step index q' = -1..L (planes L-1, 0..L-1, 0) in slot
// (q'+1) mod 5.  Every load is issued two steps before its first use.
constexpr int kSlots = 9;  // half-plane buffers per streamed path: 4 for colour 0, 5 for colour 1

template <typename Real>
struct StreamLayout {
  static __host__ __device__ int hps(int L) {  // padded half-plane, in Reals
    const int bytes = (3 * (L * L / 2) * static_cast<int>(sizeof(Real)) + 15) / 16 * 16;
    return bytes / static_cast<int>(sizeof(Real));
  }
};

// kL > 0: the lattice size is the compile-time constant kL, which turns the
// in-plane index arithmetic and the buffer offsets into immediates; kL = 0:
// any even L (sy.L).  kRS > 0: tp = kRS * L/2 threads per path, so every
// thread owns exactly kL / kRS rows at compile-time offsets.
template <typename Real, int kL, int kRS>
__device__ void run_path_streamed(const DevSystem& sy, int sys_idx, int64_t path,
                                  const SweepParams& P, unsigned char* slice, int tid, int tp,
                                  int bar, Real* lat_cta) {
  const int L = kL > 0 ? kL : sy.L, HL = L / 2, HP = L * L / 2;
  const int hps = StreamLayout<Real>::hps(L);
  const uint32_t bytes = static_cast<uint32_t>(hps * sizeof(Real));
  // [9 mbarriers][9 load counters] in 128 bytes, then the 9 half-plane buffers
  uint64_t* mbar = reinterpret_cast<uint64_t*>(slice + slice_spin_offset(tp, sy.ring, kRedBytes));
  uint32_t* issued = reinterpret_cast<uint32_t*>(mbar + kSlots);
  Real* buf = reinterpret_cast<Real*>(slice + slice_spin_offset(tp, sy.ring, kRedBytes) + 128);
  // a resumable run keeps the path's lattice in its state; otherwise the
  // group's own HBM buffer holds it for the run
  unsigned char* st = path_state(P, sys_idx, path);
  Real* lat = st ? reinterpret_cast<Real*>(st + kStateHeader) : lat_cta;
  auto plane = [&](int z, int c) { return lat + (static_cast<int64_t>(z) * 2 + c) * hps; };
  auto wrap = [&](int q) { return ((q % L) + L) % L; };
  const uint32_t c2 = static_cast<uint32_t>(sy.path_begin + path);  // path id
  const uint32_t c3u = kTagUpdate | (static_cast<uint32_t>(sys_idx) << 8);
  const uint32_t c3i = kTagInit | (static_cast<uint32_t>(sys_idx) << 8);
  const int init = path_init_mode(P.init_mode, path, sy.n_paths);
  const Real J = static_cast<Real>(sy.J), hf = static_cast<Real>(sy.h);
  const Couplings<Real> cp(P.systems + sys_idx);
  const int64_t j_first = P.s_begin > P.n_therm ? P.s_begin - P.n_therm : 0;
  Meter<Real> meter{reinterpret_cast<double*>(slice + slice_acc_offset()),
                    reinterpret_cast<Real*>(slice + slice_red_offset()),
                    sy.ring, tp >> 5, tid & 31, tid >> 5, tid,
                    1.0 / static_cast<double>(sy.N), J, hf, j_first};
  meter.start();
  __shared__ int abort_flag[kMaxGroups];  // per thread group: a bounded wait gave up, or canceled
  const int gidx = bar - 1;
  // Two threads move the half-planes, of different warps where there are two
  // (a step's copies and waits are some hundred serial cycles that the warp's
  // other work waits for): producer 0 colour 0, ring slots 0 .. 3, producer 1
  // colour 1, slots 4 .. 8.
  const int producer = tid == 0 ? 0 : tid == (tp > 32 ? 32 : 1) ? 1 : -1;
  uint32_t phases = 0;  // a producer's next wait parity of each slot
  const bool resume = P.resume && st;
  const double accepted_before = resume ? reinterpret_cast<const double*>(st)[kAccDoubles] : 0.0;

  // In-plane thread layout: column hx, rows y0, y0 + RS, ...
  const int RS = kRS > 0 ? kRS : tp / HL;
  const bool active = tid < HL * RS;
  const int hx = active ? tid % HL : 0;
  const int y0 = active ? tid / HL : L;
  // f(half-plane, half index, site index) for this thread's sites, plane by plane
  auto for_sites = [&](auto&& f) {
    for (int z = 0; z < L; ++z) {
      for (int c = 0; c < 2; ++c) {
        Real* hpl = plane(z, c);
#pragma unroll 4
        for (int y = y0; y < L; y += RS) {
          const int hp = hx + HL * y;
          f(hpl, hp, 2 * (hp + HP * z) + ((y + z + c) & 1));
        }
      }
    }
  };

  // Initial state straight into HBM (generic stores), visible to the bulk copies.
  const int N = sy.N;
  if (!resume)
    for_sites([&](Real* hpl, int hp, int i) {
      const V3<Real> v = initial_spin<Real>(static_cast<uint32_t>(i), c2, c3i, P, init);
      SpinView<Real>(hpl, HP).st(hp, v.x, v.y, v.z);
    });
  // Between calls the state holds doubles: the FP64 form's integers while a
  // call runs, each half-plane converted in place.
  auto convert_state = [&](auto&& f) {
    if constexpr (sizeof(Real) == 8) {
      for (int k = tid; k < 2 * L * 3 * HP; k += tp) f(lat + static_cast<int64_t>(k / (3 * HP)) * hps + k % (3 * HP));
    }
  };
  auto to_stored = [](Real* w) { *reinterpret_cast<typename Stored<Real>::C*>(w) = Stored<Real>::from(*w); };
  auto to_real = [](Real* w) { *w = Stored<Real>::real(*reinterpret_cast<typename Stored<Real>::C*>(w)); };
  if (resume) convert_state(to_stored);
  fence_async_global();
  if (tid < kAccDoubles) meter.acc[tid] = resume ? reinterpret_cast<const double*>(st)[tid] : 0.0;
  if (tid == 0) abort_flag[gidx] = 0;
  if (tid == 0) {
    for (int k = 0; k < kSlots; ++k) {
      mbar_init(mbar + k, 1);
      issued[k] = 0;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  auto load = [&](const Real* src, int slot) {  // the slot's producer only
    ++issued[slot];
    tma_load(buf + slot * hps, src, bytes, mbar + slot);
  };
  // every load is waited for once, in the order of the loads of its slot
  auto wait_load = [&](int slot) {
    if (!mbar_wait(mbar + slot, (phases >> slot) & 1u, P.error)) abort_flag[gidx] = 1;
    phases ^= 1u << slot;
  };
  group_sync(tp, bar);

  constexpr bool kFixedRows = kL > 0 && kRS > 0 && kL % kRS == 0;
  // FP32 with between three and four rows per thread (the planner's layouts): see phase
  constexpr bool kFourRows = sizeof(Real) == 4 && kRS == 0;
  const bool four_rows = stream_four_rows(L, RS);
  const int hp0 = hx + HL * y0;
  const StreamRows srows = stream_rows(L, RS, y0);
  int accepted = 0;
  bool ok = true;

  for (int64_t s = P.s_begin; s < P.s_end && ok; ++s) {
    const uint32_t sw = static_cast<uint32_t>(s);
    const PhiloxPrefix pre = philox_prefix(sw, c2, c3u, P.key);
    const bool meas = s >= P.n_therm;
    const int64_t j = s - P.n_therm;
    Partials<Real> part;
    // Buffers first used at step q: colour-0 index q, colour-1 index q+1 (at
    // q = 0 also colour-1 indices -1 and 0).  Only the producers wait on their
    // mbarriers; the group barrier after the wait hands the data to everyone.
    int cancel = 0;
    poll_cancel(P, s, tid, &cancel);
    if (cancel) abort_flag[gidx] = 1;  // (thread 0) stop before the sweep's first update
    if (producer == 0 && !cancel) {
      tma_wait_all();  // the previous sweep's write-backs of this colour are complete
      if (!(P.test_stall && s == P.s_begin)) load(plane(0, 0), 0);
      load(plane(1, 0), 1);
      wait_load(0);
    } else if (producer == 1) {
      tma_wait_all();
      for (int q1 = -1; q1 <= 2; ++q1) load(plane(wrap(q1), 1), 4 + q1 + 1);
      for (int k = 4; k <= 6; ++k) wait_load(k);
    }
    group_sync(tp, bar);
    if (abort_flag[gidx]) {
      ok = false;
      break;
    }
    // One colour phase over plane z: own, same-plane, +z and -z buffers.  The
    // thread's column hx is fixed, so its +-x offsets for either parity of x
    // are too (oxp1: +x when x is odd, oxm0: -x when x is even).
    const int oxp1 = (hx == HL - 1) ? -(HL - 1) : 1;
    const int oxm0 = (hx == 0) ? (HL - 1) : -1;
    auto phase = [&](int c, int z, Real* own_base, Real* same_base, Real* up_base, Real* dn_base,
                     bool energy) {
      const SpinView<Real> own(own_base, HP), same(same_base, HP), up(up_base, HP), dn(dn_base, HP);
      auto row = [&](int y) {
        const int hp = hx + HL * y;
        const int p = (y + z + c) & 1;
        const int xp = hp + (p ? oxp1 : 0);
        const int xm = hp + (p ? 0 : oxm0);
        const int yp = (y == L - 1) ? hp - (L - 1) * HL : hp + HL;
        const int ym = (y == 0) ? hp + (L - 1) * HL : hp - HL;
        const V3<Real> f = add3(add3(add3(add3(add3(same.ld(xp), same.ld(xm)), same.ld(yp)), same.ld(ym)),
                                     up.ld(hp)), dn.ld(hp));
        const uint32_t i = static_cast<uint32_t>(2 * (hp + HP * z) + p);
        if (meas) {
          if (energy)
            update<true, true>(i, pre, P.key, own, hp, f, cp, accepted, part);
          else
            update<true, false>(i, pre, P.key, own, hp, f, cp, accepted, part);
        } else {
          update<false, false>(i, pre, P.key, own, hp, f, cp, accepted, part);
        }
      };
      if constexpr (kFixedRows) {
        if (active) {
          // Rows y0 + k kRS: the x parity of row k is that of row 0 flipped
          // when k kRS is odd, and only the first row can be row 0 and only
          // the last row L - 1, so parity, x offset and the y wraps are fixed
          // at compile time for all but those.
          constexpr int kRows = kL / kRS;
          const int pz = (y0 + z + c) & 1;
          const int xoa = pz ? oxp1 : oxm0, xob = pz ? oxm0 : oxp1;
          auto rows = [&](auto meas_c, auto energy_c) {
#pragma unroll
            for (int k = 0; k < kRows; ++k) {
              const int y = y0 + k * kRS;
              const bool flip = ((k * kRS) & 1) != 0;
              const int p = flip ? pz ^ 1 : pz;
              const int hp = hx + HL * y;
              const int xo = hp + (flip ? xob : xoa);
              const int yp = (k == kRows - 1 && y == L - 1) ? hp - (L - 1) * HL : hp + HL;
              const int ym = (k == 0 && y == 0) ? hp + (L - 1) * HL : hp - HL;
              // the two x neighbours in either order (a + b = b + a exactly)
              const V3<Real> f = add3(add3(add3(add3(add3(same.ld(hp), same.ld(xo)), same.ld(yp)), same.ld(ym)),
                                           up.ld(hp)), dn.ld(hp));
              const uint32_t i = static_cast<uint32_t>(2 * (hp + HP * z) + p);
              update<decltype(meas_c)::value, decltype(energy_c)::value>(i, pre, P.key, own, hp, f, cp, accepted, part);
            }
          };
          // no branch between the rows: their Philox chains are interleaved
          if (!meas) rows(std::false_type{}, std::false_type{});
          else if (energy) rows(std::true_type{}, std::true_type{});
          else rows(std::true_type{}, std::false_type{});
        }
      } else if (kFourRows && four_rows) {
        if constexpr (kFourRows) {
          if (!active) return;
          // Rows y0 + k RS, k = 0 .. 3, the fourth only where it lies in the
          // lattice (act; stream_row): offsets, parities and wraps once per thread, no
          // branch between the rows, whose Philox chains the compiler interleaves.
          const int pz = (y0 + z + c) & 1;
          const int xoa = pz ? oxp1 : oxm0, xob = pz ? oxm0 : oxp1;
          const int xoc = (RS & 1) ? xob : xoa, pc = (RS & 1) ? pz ^ 1 : pz;
          auto rows = [&](auto meas_c, auto energy_c) {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const StreamRow row = stream_row(srows, HL, RS, k);
              const int hp = hp0 + row.off;
              const int xo = hp + (k & 1 ? xoc : xoa), p = k & 1 ? pc : pz;
              const int yp = hp + row.yp, ym = hp + row.ym;
              const V3<Real> f = add3(add3(add3(add3(add3(same.ld(hp), same.ld(xo)), same.ld(yp)), same.ld(ym)),
                                           up.ld(hp)), dn.ld(hp));
              update_spin<decltype(meas_c)::value, decltype(energy_c)::value>(
                  static_cast<uint32_t>(2 * (hp + HP * z) + p), pre, P.key, own, hp, own.ld(hp), f, cp, row.act, accepted,
                  part);
            }
          };
          if (!meas) rows(std::false_type{}, std::false_type{});
          else if (energy) rows(std::true_type{}, std::true_type{});
          else rows(std::true_type{}, std::false_type{});
        }
      } else {
#pragma unroll 4
        for (int y = y0; y < L; y += RS) row(y);
      }
    };
    // One barrier per step.  A thread updates the same half indices hp in
    // both phases, and the colour-1 site at (hp, plane q-1) has the colour-0
    // site at (hp, plane q) as its +z neighbour: phase (b) reads the thread's
    // own results of phase (a), and every other value either phase reads was
    // written before the previous barrier (in-plane neighbours of the other
    // colour come from the previous step) or is written after the next one.
    // the buffers of colour-0 indices q-2, q-1, q and colour-1 indices q-1, q, q+1
    Real *const end0 = buf + 4 * hps, *const end1 = buf + 9 * hps;
    Real *p0m2 = buf + 2 * hps, *p0m1 = buf + 3 * hps, *p0 = buf;
    Real *p1m1 = end0, *p1 = end0 + hps, *p1p1 = end0 + 2 * hps;
    int next0 = 2, next1 = 4 + 4;  // slots of the loads issued after a step: colour-0 index q+2, colour-1 index q+3
    for (int q = 0; q <= L + 1; ++q) {
      if (q < L) phase(0, q, p0, p1, p1p1, p1m1, false);
      if (q >= 2) phase(1, q > L ? 0 : q - 1, p1m1, p0m1, p0, p0m2, meas);
      fence_async_shared();
      // the buffers step q+1 starts with were issued at step q-1: their
      // producer confirms them now, and the barrier below hands them to every
      // thread
      if (producer == 0 && q <= L) wait_load((q + 1) & 3);
      if (producer == 1 && q + 1 < L) wait_load(next1 == 4 ? 8 : next1 - 1);  // colour-1 index q+2
      group_sync(tp, bar);
      if (abort_flag[gidx]) {
        ok = false;
        break;
      }
      if (meas && q == 0) meter.maybe_flush(j);
      // After the barrier the buffers just written are complete.  The slot
      // refilled now last held colour-0 index q-2 (stored after step q-2), or
      // colour-1 index q-2 (stored after step q-1): all but this step's store
      // must have finished reading shared memory.
      if (producer == 0) {
        if (q < L) tma_store(plane(q, 0), p0, bytes);
        tma_wait_read(1);
        // colour-0 step indices L and L+1 reload planes 0 and 1 written this sweep
        if (q + 2 >= L) tma_wait_all();
        if (q + 2 <= L + 1) load(plane(q + 2 >= L ? q + 2 - L : q + 2, 0), next0);
      } else if (producer == 1) {
        if (q >= 2) tma_store(plane(q > L ? 0 : q - 1, 1), p1m1, bytes);
        tma_wait_read(1);
        if (q + 3 <= L) load(plane(q + 3 == L ? 0 : q + 3, 1), next1);
      }
      next0 = (next0 + 1) & 3;
      next1 = next1 == 8 ? 4 : next1 + 1;
      p0m2 = p0m1;
      p0m1 = p0;
      p0 = p0 + hps == end0 ? buf : p0 + hps;
      p1m1 = p1;
      p1 = p1p1;
      p1p1 = p1p1 + hps == end1 ? end0 : p1p1 + hps;
    }
    if (!ok) break;
    if (meas) {
      meter.record(part);
      group_sync(tp, bar);
    }
  }
  if (producer >= 0) {
    const int k0 = producer == 0 ? 0 : 4, k1 = producer == 0 ? 4 : kSlots;
    if (!ok) {
      // a load did not arrive in time: wait (bounded) for every load still
      // in flight before the shared memory is given up
      for (int k = k0; k < k1; ++k)
        if (issued[k] > 0) mbar_wait(mbar + k, (issued[k] - 1) & 1, P.error);
    }
    tma_wait_all();
    fence_async_global();
    // every wait on them was before the last barrier, or just above
    for (int k = k0; k < k1; ++k) mbar_inval(mbar + k);
  }
  group_sync(tp, bar);
  if (!ok) {  // the error flag is set; the path's record is not written
    if (st) convert_state(to_real);
    return;
  }
  const int64_t n_meas_done = P.s_end > P.n_therm ? P.s_end - P.n_therm : 0;
  meter.finish(n_meas_done);
  group_sync(tp, bar);

  Real worst = Real(0);  // in the working precision: FP64 runs at 1/64 rate on this GPU
  if (P.spins == nullptr) {
    for_sites([&](Real* hpl, int hp, int) { worst = fmax(worst, norm_error(SpinView<Real>(hpl, HP).ld(hp))); });
  } else {
    double* out = P.spins + P.spin_offset[sys_idx] + path * 3 * static_cast<int64_t>(N);
    for_sites([&](Real* hpl, int hp, int i) {
      const V3<Real> v = SpinView<Real>(hpl, HP).ld(hp);
      worst = fmax(worst, norm_error(v));
      out[3 * i + 0] = Stored<Real>::real(v.x);
      out[3 * i + 1] = Stored<Real>::real(v.y);
      out[3 * i + 2] = Stored<Real>::real(v.z);
    });
  }
  if (st) {
    group_sync(tp, bar);  // every spin has been read
    convert_state(to_real);
  }
  if (P.save && st && tid < kAccDoubles) reinterpret_cast<double*>(st)[tid] = meter.acc[tid];
  meter.write_record(P.records + (sy.rec_offset + path) * MP_NREC, accepted,
                     static_cast<double>(worst), P.s_end, n_meas_done, N, tp, bar, accepted_before,
                     (P.save && st) ? reinterpret_cast<double*>(st) + kAccDoubles : nullptr);
  group_sync(tp, bar);  // the slice and the HBM buffer are reused by the next item
}

// ------------------------------------------------------- persistent loop --
// The compile-time lattice sizes each precision supports in shared memory.
#define MPK_FOR_EACH_L_FP32(X) X(2) X(4) X(6) X(8) X(10) X(12) X(14) X(16) X(18) X(20) X(22) X(24) X(26)
#define MPK_FOR_EACH_L_FP64(X) X(2) X(4) X(6) X(8) X(10) X(12) X(14) X(16) X(18) X(20)

// Kernel variants: kLattice > 0 runs only simple cubic L = kLattice (a batch of
// one size), kLattice = kChainKernel only open chains, kLattice = kMixedKernel
// switches on each work item's lattice (a batch of uneven sizes).
constexpr int kMixedKernel = 0;
constexpr int kChainKernel = -1;
constexpr int kChainOneKernel = -6;  // chains with a thread for every site of a colour
constexpr int kStreamKernel = -2;  // simple cubic lattices streamed from HBM (any even L)
// simple cubic lattices of one size L streamed from HBM, compiled for that L
__host__ __device__ constexpr int stream_variant(int L) { return -1000 - L; }
__host__ __device__ constexpr int stream_variant_L(int v) { return v <= -1000 ? -1000 - v : 0; }

template <typename Real, int kLattice>
__device__ __forceinline__ void dispatch_path(const DevSystem& sy, int sys_idx, int64_t path,
                                              const SweepParams& P, unsigned char* slice, int tid,
                                              int tp, int bar);

// Largest CTA of every sweep kernel: 512 threads with up to 128 registers per
// thread, which the FP64 form needs and which buys the FP32 column walk its
// unrolled instruction-level parallelism.  (1024-thread CTAs at 64 registers
// were measured 6-16% slower for L = 18 and 24.)
// Two CTAs per SM (64 registers) where a lane has one site per half-sweep and
// little to interleave: FP32 L <= 4 (one-site form, L = 4 with 40000 paths 1.27e11
// -> 1.8e11 attempts/s; FP64 chains too take that form) and FP32 chains (64 spins,
// 90112 paths 1.31e11 -> 1.67e11; there the one-site form gave 1.44e11, and chains
// with more sites per lane lose 10% to the shorter register file).
template <typename Real, int kLattice>
constexpr bool kOneSite = kLattice == 2 || kLattice == 4 || (sizeof(Real) == 8 && kLattice == kChainOneKernel);
template <typename Real, int kLattice>
struct CtaLimit {
  static constexpr int value = 512;
  static constexpr int per_sm =
      sizeof(Real) == 4 && (kLattice == 2 || kLattice == 4 || kLattice == kChainOneKernel) ? 2 : 1;
};

template <typename Real, int kLattice>
__global__ void __launch_bounds__(CtaLimit<Real, kLattice>::value, CtaLimit<Real, kLattice>::per_sm)
    sweep_kernel(const SweepParams P) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ int s_item;
  if constexpr (sizeof(Real) == 8) {  // read after the first barrier below
    for (int k = static_cast<int>(threadIdx.x); k < 256; k += static_cast<int>(blockDim.x))
      sine_shared()[k] = kSineTable.s[k];
  }
  if constexpr (kLattice == kMixedKernel && sizeof(Real) == 4) {
    // First the lattices held by two CTAs: the cluster takes one path at a
    // time from its own queue (rank 0 draws, both CTAs read), then each CTA
    // goes on to the single-CTA items below.
    if (P.n_pair_items > 0) {
      if (cluster_size() != 2) {
        if (threadIdx.x == 0) atomicExch(P.error, kErrLaunch);
      } else {
        __shared__ int s_pair;
        const uint32_t rank = cluster_rank();
        for (;;) {
          if (rank == 0 && threadIdx.x == 0) {
            const int it = atomicAdd(P.pair_queue, 1);
            s_pair = it;
            *map_rank(&s_pair, 1u) = it;
          }
          cluster_sync_all();
          const int item = s_pair;
          cluster_sync_all();  // both CTAs have read the item before rank 0 draws again
          if (item >= P.n_pair_items) break;
          const WorkItem it = P.pair_items[item];
          run_path_pair<Real, kPairL>(P.systems[it.sys], it.sys, it.path0, P, smem,
                                      static_cast<int>(threadIdx.x), static_cast<int>(blockDim.x), rank);
        }
      }
    }
  }
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
    if (g < it.count) {
      bool done = false;
      if constexpr (stream_variant_L(kLattice) > 0) {
        Real* lat = reinterpret_cast<Real*>(
            static_cast<unsigned char*>(P.lattice) +
            (static_cast<int64_t>(blockIdx.x) * P.lattice_groups + g) * P.lattice_stride);
        constexpr int kL = stream_variant_L(kLattice);
        if (sy.tp == 8 * kL)  // 16 row groups of L/2 threads: L/16 rows per thread
          run_path_streamed<Real, kL, 16>(sy, it.sys, it.path0 + g, P, smem + g * sy.slice_bytes,
                                          tid, sy.tp, 1 + g, lat);
        else if (sy.tp == 4 * kL)  // 8 row groups: L/8 rows per thread
          run_path_streamed<Real, kL, 8>(sy, it.sys, it.path0 + g, P, smem + g * sy.slice_bytes,
                                         tid, sy.tp, 1 + g, lat);
        else
          run_path_streamed<Real, kL, 0>(sy, it.sys, it.path0 + g, P, smem + g * sy.slice_bytes,
                                         tid, sy.tp, 1 + g, lat);
        done = true;
      }
      if constexpr (kLattice == kStreamKernel || kLattice == kMixedKernel || kLattice == kGlobalKernel) {
        if (!done && sy.mode == kModeGlobal) {
          Real* lat = reinterpret_cast<Real*>(
              static_cast<unsigned char*>(P.lattice) +
              (static_cast<int64_t>(blockIdx.x) * P.lattice_groups + g) * P.lattice_stride);
          run_path<Real>(GeomSCDyn{sy.L}, sy, it.sys, it.path0 + g, P, smem + g * sy.slice_bytes, tid,
                         sy.tp, 1 + g, lat);
          done = true;
        }
      }
      if constexpr (kLattice == kStreamKernel || kLattice == kMixedKernel) {
        if (!done && sy.mode == kModeStreamed) {
          Real* lat = reinterpret_cast<Real*>(
              static_cast<unsigned char*>(P.lattice) +
              (static_cast<int64_t>(blockIdx.x) * P.lattice_groups + g) * P.lattice_stride);
          if constexpr (kLattice == kMixedKernel) {
            // batches of uneven sizes: the streamed size of the benchmark's
            // batch (L = 32) with compile-time rows
            if (sy.L == 32 && sy.tp == 8 * 32)
              run_path_streamed<Real, 32, 16>(sy, it.sys, it.path0 + g, P, smem + g * sy.slice_bytes,
                                              tid, sy.tp, 1 + g, lat);
            else if (sy.L == 32 && sy.tp == 4 * 32)
              run_path_streamed<Real, 32, 8>(sy, it.sys, it.path0 + g, P, smem + g * sy.slice_bytes,
                                             tid, sy.tp, 1 + g, lat);
            else
              run_path_streamed<Real, 0, 0>(sy, it.sys, it.path0 + g, P, smem + g * sy.slice_bytes,
                                            tid, sy.tp, 1 + g, lat);
          } else {
            run_path_streamed<Real, 0, 0>(sy, it.sys, it.path0 + g, P, smem + g * sy.slice_bytes, tid,
                                          sy.tp, 1 + g, lat);
          }
          done = true;
        }
      }
      if (!done)
        dispatch_path<Real, kLattice>(sy, it.sys, it.path0 + g, P, smem + g * sy.slice_bytes, tid,
                                      sy.tp, 1 + g);
    }
  }
}

}  // namespace mpk
