// The FP64 form's spins as 64-bit fixed point.
//
// GB300 issues one FP64 warp instruction per scheduler every 76 cycles (FP64
// add, multiply and fused multiply-add alike), but a 64-bit integer add costs
// 2.5 cycles and a 32 x 32 -> 64 multiply 4.  A spin component of the FP64
// form is therefore kept as an integer multiple of 2^-53 in [-2^53, 2^53]:
// every such number is a double, so records, spins and saved states hold it
// exactly, and it lies as close to the real value as a double in [1/2, 1)
// can.  Sums of spins (local fields, magnetisation) are then exact integer
// sums, with no rounding at all, in any order.
//
// The trial direction (cos(theta) = 2 u0 - 1, phi = 2 pi u1 for u = (r + 1/2)
// 2^-32) is evaluated in 63-bit fixed point from the two words: the square root
// by two Newton steps from the hardware's FP32 reciprocal square root with
// exact integer residuals, sine and cosine by the angle-addition formulas
// around 256 table points per quarter turn and Taylor terms of the remainder.
// Over 3e6 pairs of words, edges included, a component is off by at most
// 2^-53.7 and 3.2e-17 rms, the rounding to the grid; double sqrt and sincos of
// the rounded 2 pi u1 gave 2^-50.4 and 7.8e-17.
#pragma once
#include <cmath>
#include <cstdint>

namespace mpk {

constexpr int kFixBits = 53;  // fraction bits of a spin component

#ifdef __CUDA_ARCH__
#define MPK_UMULHI(a, b) __umulhi(a, b)
#define MPK_RSQRT(x) rsqrtf(x)
#define MPK_F2I(x) __float2int_rn(x)
#define MPK_F2U(x) __float2uint_rz(x)
#else
// Host forms of the same steps, for the accuracy test.
inline uint32_t mpk_host_umulhi(uint32_t a, uint32_t b) {
  return static_cast<uint32_t>((static_cast<uint64_t>(a) * b) >> 32);
}
#define MPK_UMULHI(a, b) mpk_host_umulhi(a, b)
#define MPK_RSQRT(x) (1.0f / std::sqrt(x))
#define MPK_F2I(x) static_cast<int32_t>(std::lrint(x))
#define MPK_F2U(x) ((x) >= 4294967296.0f ? 0xffffffffu : static_cast<uint32_t>(x))
#endif

// sin((pi/2) (j + 1/2) / 256) in units of 2^-63, j = 0 .. 255 (the cosine of
// point j is the sine of point 255 - j), from the Taylor series in integers.
struct SineTable {
  uint64_t s[256];
};
constexpr uint64_t mul_shift62(uint64_t a, uint64_t b) {
  return static_cast<uint64_t>((static_cast<unsigned __int128>(a) * b + (static_cast<unsigned __int128>(1) << 61)) >> 62);
}
constexpr SineTable make_sine_table() {
  SineTable t{};
  // pi/2 in units of 2^-62: floor(pi 2^61)
  constexpr uint64_t kHalfPi62 = 0x6487ED5110B4611Aull;
  for (int j = 0; j < 256; ++j) {
    // x = (pi/2) (2 j + 1) / 512 < pi/2 in units of 2^-62
    const uint64_t x =
        static_cast<uint64_t>((static_cast<unsigned __int128>(kHalfPi62) * (2 * j + 1) + 256) >> 9);
    const uint64_t x2 = mul_shift62(x, x);  // < 2.47 < 4
    uint64_t term = x, pos = x, neg = 0;
    for (int k = 1; k < 16 && term > 0; ++k) {
      const uint64_t d = static_cast<uint64_t>(2 * k) * (2 * k + 1);
      term = (mul_shift62(term, x2) + d / 2) / d;
      if (k & 1) neg += term;
      else pos += term;
    }
    t.s[j] = (pos - neg) << 1;
  }
  return t;
}

// High 64 bits of a 64 x 64-bit product without its low x low part (at most 2
// units below the exact value).
__host__ __device__ __forceinline__ uint64_t mulhi_short(uint64_t a, uint64_t b) {
  const uint32_t ah = static_cast<uint32_t>(a >> 32), al = static_cast<uint32_t>(a);
  const uint32_t bh = static_cast<uint32_t>(b >> 32), bl = static_cast<uint32_t>(b);
  return static_cast<uint64_t>(ah) * bh + MPK_UMULHI(ah, bl) + MPK_UMULHI(al, bh);
}

// A 64-bit integer as a float (two conversions, relative error 2^-23).
__host__ __device__ __forceinline__ float fix_float(int64_t v) {
  return static_cast<float>(static_cast<int32_t>(v >> 32)) * 4294967296.0f +
         static_cast<float>(static_cast<uint32_t>(v));
}

struct Fix3 {
  int64_t x, y, z;
};

// cos(theta) = 2 u0 - 1 for the word r0, exactly.
__host__ __device__ __forceinline__ int64_t fix_cos_theta(uint32_t r0) {
  const int64_t w = (static_cast<int64_t>(r0) * 2 + 1) - (int64_t{1} << 32);  // z 2^32
  return w * (int64_t{1} << (kFixBits - 32));
}

// 1 - z^2 for the word r0: n = 2^64 (1 - z^2), an exact 64-bit integer (z 2^32 is
// an odd integer below 2^32 in magnitude), and y = 1/sqrt(n) from the hardware.
struct FixRoot {
  uint64_t n;
  float nf, y;
};
__host__ __device__ __forceinline__ FixRoot fix_root(uint32_t r0) {
  const uint32_t wm = (r0 & 0x80000000u) ? r0 * 2u + 1u : ~(r0 * 2u + 1u) + 1u;  // |z| 2^32
  FixRoot q;
  q.n = uint64_t{0} - static_cast<uint64_t>(wm) * wm;
  q.nf = static_cast<float>(static_cast<uint32_t>(q.n >> 32)) * 4294967296.0f +
         static_cast<float>(static_cast<uint32_t>(q.n));
  q.y = MPK_RSQRT(q.nf);
  return q;
}

// The trial direction of the words r0, r1 with q = fix_root(r0); `sine` is the
// table above.
__host__ __device__ __forceinline__ Fix3 fix_trial(uint32_t r0, uint32_t r1, const FixRoot& q,
                                                   const uint64_t* sine) {
  // rad = sqrt(n), in units of 2^-63 of 2^32
  const float hy = 0.5f * q.y;
  const uint32_t s0 = MPK_F2U(q.nf * q.y);  // sqrt(n) to 2^-21
  const int64_t e1 = static_cast<int64_t>(q.n - static_cast<uint64_t>(s0) * s0);
  const int64_t c1 = MPK_F2I(fix_float(e1) * hy * 65536.0f);
  const uint64_t t1 = (static_cast<uint64_t>(s0) << 16) + static_cast<uint64_t>(c1);  // sqrt(n) 2^16 to 2^-42
  const int64_t e2 = static_cast<int64_t>((q.n << 32) - t1 * t1);  // small: the difference modulo 2^64 is exact
  const uint64_t rad = (t1 << 15) + static_cast<uint64_t>(static_cast<int64_t>(MPK_F2I(fix_float(e2) * hy * 0.5f)));

  // phi = 2 pi (2 r1 + 1) / 2^33: quarter turn, table point j and the offset
  // d = (pi/2) dr / 2^31 from it, |d| <= pi/1024
  const uint32_t quarter = r1 >> 30;
  const uint32_t rem = (r1 << 1 | 1u) & 0x7fffffffu;  // 31-bit fraction of the quarter turn
  const uint32_t j = rem >> 23;
  const int32_t dr = static_cast<int32_t>(rem & 0x7fffffu) - 0x400000;
  const uint32_t da = static_cast<uint32_t>(dr < 0 ? -dr : dr);
  // |d| in units of 2^-64: da (pi/2) 2^33, pi/2 2^63 = 0xC90FDAA22168C235
  const uint64_t d = (static_cast<uint64_t>(da) * 0xC90FDAA2u << 2) + (static_cast<uint64_t>(da) * 0x2168C235u >> 30);
  const uint32_t dh = static_cast<uint32_t>(d >> 24), dl = static_cast<uint32_t>(d) & 0xffffffu;
  const uint64_t d2 = static_cast<uint64_t>(dh) * dh + (static_cast<uint64_t>(dh) * dl >> 23);  // d^2, 2^-80
  const uint32_t d2h = static_cast<uint32_t>(d2 >> 32);                                         // d^2, 2^-48
  const uint32_t d4 = MPK_UMULHI(d2h, d2h);                                                     // d^4, 2^-64
  const uint64_t ver = (d2 >> 17) - MPK_UMULHI(d4, 0x0AAAAAABu);        // 1 - cos d = d^2/2 - d^4/24, 2^-64
  const uint32_t w6 = MPK_UMULHI(d2h, 0x2AAAAAABu) - (MPK_UMULHI(d4, 0x02222222u) >> 16);  // d^2/6 - d^4/120, 2^-48
  const uint64_t sn = d - (static_cast<uint64_t>(dh) * w6 >> 24);       // sin |d|, 2^-64
  const uint64_t S = sine[j], C = sine[255u - j];
  const uint64_t cs = mulhi_short(C, sn), ss = mulhi_short(S, sn);
  // sin(a + d), cos(a + d), units of 2^-63
  const uint64_t sv = S - mulhi_short(S, ver), cv = C - mulhi_short(C, ver);
  const uint64_t sa = dr < 0 ? sv - cs : sv + cs;
  const uint64_t ca = dr < 0 ? cv + ss : cv - ss;

  // components of magnitude rad cos, rad sin, rounded to the 2^-53 grid
  const int64_t a = static_cast<int64_t>((mulhi_short(rad, ca) + 256u) >> 9);
  const int64_t b = static_cast<int64_t>((mulhi_short(rad, sa) + 256u) >> 9);
  Fix3 t;
  const int64_t px = (quarter & 1u) ? b : a, py = (quarter & 1u) ? a : b;
  t.x = (quarter == 1u || quarter == 2u) ? -px : px;
  t.y = (quarter & 2u) ? -py : py;
  t.z = fix_cos_theta(r0);
  return t;
}

}  // namespace mpk
