// Standard normals from counter blocks: Philox4x32-10 words and Box-Muller in
// 64-bit fixed point.
//
// GB300 issues a float64 warp instruction every 64 cycles of a scheduler and a
// 64-bit high product every ~30, so the logarithm and the sine and cosine, which
// are polynomials on a bounded range, are summed in integers (the logarithm after
// Tang's table-driven method, ACM TOMS 16, 1990); what is left on the
// float64 pipe is a pair's one multiply-add, root and two products.  Their inputs
// are exact: u = (x + 1/2) 2^-32 is an odd integer over 2^33.
// Against 113-bit arithmetic, three million pairs with the ends of the range: a
// normal's error 9.6e-17 rms, 1.5e-15 at most (float64 log, sqrt and sincos of the
// rounded 2 pi u: 2.8e-16 and 4.5e-15).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

namespace pycool {

// high 64 bits of a 64 x 64-bit signed product
__host__ __device__ __forceinline__ long long mul_hi(long long a, long long b) {
#ifdef __CUDA_ARCH__
  return __mul64hi(a, b);
#else
  return (long long)(((__int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ int lead_zeros(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}
// x 2^-s, |x| < 2^63, rounded to nearest (a tie away from zero), in integers: the
// conversion instruction runs at the float64 rate
__host__ __device__ __forceinline__ double scaled(long long x, int s) {
  const unsigned long long a = x < 0 ? 0ull - (unsigned long long)x : (unsigned long long)x;
  if (a == 0ull) return 0.0;
  const int lz = lead_zeros(a);
  const unsigned long long m = a << lz;
  unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);
  r += (unsigned long long)(uint32_t)(1085 - s - lz) << 52;
  if (x < 0) r |= 0x8000000000000000ull;
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)r);
#else
  double d;
  __builtin_memcpy(&d, &r, 8);
  return d;
#endif
}

// ln(c_j) 2^62 of the 64 reciprocals c_j = kLogRecip[j] / 256 (j < 32) or / 128
// of the mid-points of [1 + j/64, 1 + (j + 1)/64), rounded to eight or nine bits
// so that M c_j is exact; the first and last are 1, so that nothing cancels
// beside u = 1.
#define PYCOOL_LOG_TABLE                                                                   \
  {0x0ll,                -0x18492528c8cabe9ll,  -0x28cd5da85bc7d32ll,  -0x355de5a1f621f83ll,  \
   -0x465cef4519559b4ll, -0x534c457481fab17ll,  -0x64cd7975652622cll,  -0x72216006f12c8dall,  \
   -0x7fa244e76f55965ll, -0x8d515bf11fb94f2ll,  -0x9b2fe580ac80b18ll,  -0xa93f2f250dac67dll,  \
   -0xb780945bab55dcell, -0xc5f57f59c7f4615ll,  -0xcfb6203844b320all,  -0xde8439c1dec5687ll,  \
   -0xe881bf932af3dacll, -0xf7ad6f26e7ff2efll,  -0x101eae5626c690f7ll, -0x11178e8227e47bdell, \
   -0x11bf99635a6b94dell, -0x1269621134db9278ll, -0x136b6776be1116edll, -0x1419b423d5e8c722ll, \
   -0x14c9e09e172c3befll, -0x157bf753c8d1fadfll, -0x1630030b3aac493cll, -0x16e60ee6af197216ll, \
   -0x179e26687cfb3d90ll, -0x185855776dcbfaaell, -0x1914a8635bf68995ll, -0x1973a3431356adcfll, \
   0x122941fbcf7965a2ll, 0x11675cababa60e04ll,  0x10a324e27390e35fll,  0x10402594b4d040dbll,  \
   0xf7856e5ee2c9b29ll,  0xeae10b5a7ddc8aell,   0xe47fbe3cd4d10d6ll,   0xd79e4a7405ff96cll,   \
   0xd11de0ff15ab18dll,  0xc3fd03290648848ll,   0xbd5c481086c848ell,   0xaff983853c9e9e4ll,   \
   0xa9372f1d0da1bd1ll,  0xa2695b665be8f34ll,   0x94aa97c0ffa91a6ll,   0x8db956a97b3d015ll,   \
   0x86bbf3e68472cb3ll,  0x789c1db8abcb97all,   0x7179523d6f1d0c5ll,   0x6a49b4e92b558d9ll,   \
   0x630d1758c66c83dll,  0x546c1cfc1860fdall,   0x4d075e586f47425ll,   0x4594dbba8deb83all,   \
   0x3e14618022c54ccll,  0x3685bae232e37d8ll,   0x2ee8b1ec65b9f89ll,   0x273d0f73fd7abf5ll,   \
   0x1f829b0e7833005ll,  0x17b91b07d5b11abll,   0xfe054587e01f1ell,    0x0ll}
#define PYCOOL_LOG_RECIP                                                                     \
  {256, 250, 246, 243, 239, 236, 232, 229, 226, 223, 220, 217, 214, 211, 209, 206,           \
   204, 201, 199, 196, 194, 192, 189, 187, 185, 183, 181, 179, 177, 175, 173, 172,           \
   170, 168, 166, 165, 163, 161, 160, 158, 157, 155, 154, 152, 151, 150, 148, 147,           \
   146, 144, 143, 142, 141, 139, 138, 137, 136, 135, 134, 133, 132, 131, 130, 128}

// -2 ln((2 x + 1) 2^-33).  u = M 2^e, M in [1, 2), or M/2 and e + 1 from M = 1.5
// on; ln M = ln(1 + r) - ln c_j with r = M c_j - 1 exact, |r| <= 2^-6, and
// ln(1 + r) = r P(r), P by the Taylor series to r^8 (the next term is 2^-57 of P).
__host__ __device__ __forceinline__ double minus2log(uint32_t x, const long long* table,
                                                     const int* recip) {
  const unsigned long long a = 2ull * x + 1ull;
  const int lz = lead_zeros(a);
  const unsigned long long m = a << lz;                    // M 2^63
  const int j = (int)(m >> 57) & 63;
  const int e = 30 - lz + (j >= 32 ? 1 : 0);               // <= 0
  const long long d = (long long)((m >> 8) * (unsigned long long)recip[j] - 0x8000000000000000ull);
  const long long R = d << 6;                              // r 2^69 (d is r 2^63, exact)
  long long P = 0x71c71c71c71c71cll;                       // 1/9 ... in units of 2^-62
  P = -0x800000000000000ll + (mul_hi(R, P) >> 5);
  P = 0x924924924924925ll + (mul_hi(R, P) >> 5);
  P = -0xaaaaaaaaaaaaaabll + (mul_hi(R, P) >> 5);
  P = 0xccccccccccccccdll + (mul_hi(R, P) >> 5);
  P = -0x1000000000000000ll + (mul_hi(R, P) >> 5);
  P = 0x1555555555555555ll + (mul_hi(R, P) >> 5);
  P = -0x2000000000000000ll + (mul_hi(R, P) >> 5);
  P = 0x4000000000000000ll + (mul_hi(R, P) >> 5);
  if (j == 63 && e == 0) return scaled(R, 68) * -scaled(P, 62);   // beside u = 1: relative
  const double t = scaled(table[j] - (mul_hi(R, P) >> 5), 61);    // -2 ln(M or M/2)
  return fma(scaled(-2 * e, 0), 0.6931471805599453, t);
}

// (cos, sin) of 2 pi (2 x + 1) 2^-33 in units of 2^-62: the nearest quarter turn
// and the rest y pi/4, |y| <= 1, by the Taylor series in y^2 (to y^18 and y^17:
// the next terms are below 2^-62).
__host__ __device__ __forceinline__ void turn62(uint32_t x, long long& cs, long long& sn) {
  const unsigned long long p = (2ull * x + 1ull) << 31;    // turns 2^64
  const unsigned int q = (unsigned int)((p + 0x2000000000000000ull) >> 62);
  const long long y = (long long)((p - ((unsigned long long)q << 62)) << 2);   // y 2^63
  const long long w = mul_hi(y, y);                        // y^2 2^62
  long long c = -0x9ll;
  c = 0x120cll + (mul_hi(w, c) << 2);
  c = -0x1b6e25ll + (mul_hi(w, c) << 2);
  c = 0x1f9d38a3ll + (mul_hi(w, c) << 2);
  c = -0x1a6d1f2a20ll + (mul_hi(w, c) << 2);
  c = 0xf0fa83448ddll + (mul_hi(w, c) << 2);
  c = -0x5574f1f8f2ffell + (mul_hi(w, c) << 2);
  c = 0x103c1f081b5ac3bll + (mul_hi(w, c) << 2);
  c = -0x13bd3cc9be45de5all + (mul_hi(w, c) << 2);
  c = 0x4000000000000000ll + (mul_hi(w, c) << 2);
  long long s = 0xd5ll;
  s = -0x16faell + (mul_hi(w, s) << 2);
  s = 0x1e8f435ll + (mul_hi(w, s) << 2);
  s = -0x1e3074fdfll + (mul_hi(w, s) << 2);
  s = 0x150783487eell + (mul_hi(w, s) << 2);
  s = -0x9969667315ecll + (mul_hi(w, s) << 2);
  s = 0x28cd78ceeb55c4ll + (mul_hi(w, s) << 2);
  s = -0x52aef39896f94b0ll + (mul_hi(w, s) << 2);
  s = 0x3243f6a8885a308dll + (mul_hi(w, s) << 2);
  s = mul_hi(y, s) << 1;
  const bool swap = q & 1u;
  cs = swap ? s : c;
  sn = swap ? c : s;
  if ((q + 1u) & 2u) cs = -cs;   // quarters 1 and 2
  if (q & 2u) sn = -sn;          // quarters 2 and 3
}

}  // namespace pycool
