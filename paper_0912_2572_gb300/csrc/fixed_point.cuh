// 64-bit fixed-point helpers shared by the factorization job (factor_fixed.cuh) and the
// tensor-core apply kernel (apply_mma.cu): a column is held as integers x 2^(60 - E) with
// its 2-norm below 2^60.
#pragma once
#include <cstdint>

namespace tsqr {
namespace {

constexpr int kFxNone = -100000;     // no exponent yet (no nonzero entry seen)
constexpr int kFxMaxExp = 900;       // entries of magnitude outside 2^+-900 (and non-finite ones)
                                     // go through the FP64 job

// a b + c. Written as the instruction: from (long long)a * b the compiler made full 64-bit
// products wherever the operands were halves of 64-bit registers (four times the multiplies).
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
}

// x 2^s, rounded to nearest for s < 0
__device__ __forceinline__ long long fx_shift(long long x, int s) {
  if (s >= 0) return s > 63 ? 0 : (long long)((unsigned long long)x << s);
  if (s < -62) return 0;
  return (x + (1ll << (-s - 1))) >> (-s);
}

__device__ __forceinline__ long long fx_of_double(long long bits, int sh) {  // round(x 2^sh)
  const int e = (int)((bits >> 52) & 0x7ff);
  if (e == 0 || e + sh <= 0) return 0;
  return __double2ll_rn(__longlong_as_double(bits + ((long long)sh << 52)));
}
__device__ __forceinline__ double fx_to_double(long long x, int sh) {  // x 2^sh
  const long long b = __double_as_longlong(__ll2double_rn(x));
  return __longlong_as_double(x == 0 ? 0ll : b + ((long long)sh << 52));
}

// The magnitude bits of a double's high word, and its square relative to 2^(2t) as FP32
// (20 mantissa bits), for the norm bound of a column whose largest exponent field is e (t =
// e - 1022).
__device__ __forceinline__ float fx_square_rel(unsigned habs, unsigned e) {
  const int f = (int)(habs - ((e - 126u) << 20));
  const float x = __int_as_float(f > 0 ? f << 3 : 0);
  return x * x;
}
// Adds entries of squared norm sq 2^(2t) to a column of squared norm nb 2^(2E).
__device__ __forceinline__ void fx_grow(int &E, float &nb, int t, float sq) {
  const int base = max(E, t);
  float s = sq * 1.00002f * exp2f((float)max(2 * (t - base), -140));
  if (E > kFxNone) s += nb * exp2f((float)max(2 * (E - base), -140));
  int b = base;
  while (s >= 0.9f) {
    ++b;
    s *= 0.25f;
  }
  E = b;
  nb = s;
}

// Light tiles. An entry of 2^-s of its column's norm keeps 60 - s bits here, where FP64 keeps
// 53 of every entry, and what it lost matters once the heavy rows of the column are eliminated:
// in weighted least squares with the heavy rows first (weights of 1e8 are ordinary for soft
// constraints) the light rows alone determine the rest of the unknowns. A tile is light in a
// column, and its job goes on in FP64 from there, if the root mean square of the tile's nonzero
// entries is below 2^-12 of 2^E, or more of them than a smooth distribution would have (its
// density at zero is below 1 / rms: eight times that) are below 2^-16. The rows of a chain of
// M alike rows are at 2^-(1 + log2(M) / 2), so plain chains of up to 2^22 rows stay. A node's
// triangle falls off along its rows by itself when A is ill-conditioned: there a quarter of the
// entries may be that small, and the later pieces of a triangle are not looked at. Costs two
// instructions per entry and tile, beside 37 cycles per entry and step.
constexpr int kFxLightBits = 16;
// nz entries, nl of them light, their squares' sum sq 4^d in units of the column's 4^E
__device__ __forceinline__ bool fx_light(unsigned nz, unsigned nl, float sq, int d, bool tri) {
  if (nz == 0) return false;
  const float fz = (float)nz, q = sq * exp2f((float)max(2 * d, -100)) / fz;
  return q < 0x1p-24f || (float)nl > 4.f + fz * fmaxf(0x1p-13f * rsqrtf(q), tri ? 0.25f : 0.f);
}

// ah 2^30 + al = a, al signed
__device__ __forceinline__ void fx_limbs(long long a, int &h, int &l) {
  h = (int)((a + (1ll << 29)) >> 30);
  l = (int)((unsigned)a - ((unsigned)h << 30));
}
// a b / 2^S for S = 59, 60 or 61, to within a unit
template <int S>
__device__ __forceinline__ long long fx_mul(int ah, int al, int2 b) {
  const long long m = fx_mad(ah, b.y, fx_mad(al, b.x, 1ll << (S - 31)));
  const long long h = fx_mad(ah, b.x, 0);
  if constexpr (S <= 60) return h * (1ll << (60 - S)) + (m >> (S - 30));
  else return (h + (m >> 30)) >> 1;
}

}  // namespace
}  // namespace tsqr
