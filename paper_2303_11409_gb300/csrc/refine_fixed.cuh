// Fixed-point form of the operands of the refinement's products (k_refine.cu): a column of an operand is scaled by a
// power of two, 2^e above the largest of its parts, and each part becomes the integer x 2^(54 - e) in 7 balanced
// base-256 digits.
#pragma once
#include <climits>
#include <cstdint>
#include <cstring>

namespace mps {

__host__ __device__ inline int float_bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_int(x);
#else
  int b;
  std::memcpy(&b, &x, 4);
  return b;
#endif
}
__host__ __device__ inline long long double_bits(double x) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(x);
#else
  long long b;
  std::memcpy(&b, &x, 8);
  return b;
#endif
}

// x 2^(54 - e) rounded to an integer, plus 128 in every one of the 7 low bytes (balanced digits are
// then byte - 128); |x| < 2^e.
__host__ __device__ inline uint64_t oz_fixed(double x, int e) {
  const long long b = double_bits(x);
  const int E = (int)((b >> 52) & 0x7ff);
  const long long mant = (b & 0xfffffffffffffLL) | 0x10000000000000LL;
  const int s = E - 1021 - e;
  long long q;
  if (s >= 0) q = mant << (s < 1 ? s : 1);
  else q = s < -54 ? 0 : (mant + (1LL << (-s - 1))) >> (-s);
  if (b < 0) q = -q;
  return (uint64_t)(q + 0x0080808080808080LL);
}
__host__ __device__ inline uint64_t oz_fixed(float x, int e) {
  const int b = float_bits(x);
  const int E = (b >> 23) & 0xff;
  const long long mant = (b & 0x7fffff) | 0x800000;
  const int s = E - 96 - e;      // x = mant 2^(E - 150)
  long long q;
  if (E == 0) q = 0;
  else if (s >= 0) q = mant << (s < 30 ? s : 30);
  else q = s < -25 ? 0 : (mant + (1LL << (-s - 1))) >> (-s);
  if (b < 0) q = -q;
  return (uint64_t)(q + 0x0080808080808080LL);
}

// The smallest e with |x| < 2^e (zero and denormals: below every other).
__host__ __device__ inline int exponent_above(float x) {
  const int E = (float_bits(x) >> 23) & 0xff;
  return E ? E - 126 : INT_MIN / 2;
}

// A column of the correction W of a refinement step: the entries E_kc off the diagonal, and E_cc - sq / 2 on it with
// sq = sum_k |E_kc|^2.  The diagonal is one part of the column like the others: scaled apart, as E_cc and sq, it
// could reach 1.5 times the scale when both are negative.
struct CorrectionScale {
  int top = INT_MIN / 2;
  float sq = 0.f, diag = 0.f;
  // entry k as stored, w = E_kc 2^-d; shift: the exponent that the product's other operand brings
  __host__ __device__ void add(float x, float y, int d, int shift, bool on_diagonal) {
    const float f = exp2f((float)(d < -60 ? -60 : d > 60 ? 60 : d));
    sq = fmaf(x * f, x * f, fmaf(y * f, y * f, sq));
    if (on_diagonal) {
      diag = x;
    } else {
      const int ex = exponent_above(x), ey = exponent_above(y), e = ex > ey ? ex : ey;
      if (e > INT_MIN / 2 && e + shift > top) top = e + shift;
    }
  }
  __host__ __device__ float second_order() const { return -0.5f * sq; }
  // of the whole column, once top, sq and diag are
  __host__ __device__ int scale(int shift) const {
    const int e = exponent_above(diag + second_order());
    const int t = e > INT_MIN / 2 && e + shift > top ? e + shift : top;
    return t > -1000 ? t : -1000;
  }
};

}  // namespace mps
