// Real 3-D transforms of float64 arrays in block-scaled 64-bit fixed point.
//
// A float64 transform on GB300 is bound by its float64 pipe (two lanes per SM
// and clock): a 256-point pass takes some 25 float64 instructions a point, and
// three quarters of them are additions.  Here a line of points is put on a
// common 64-bit fixed-point scale (58 bits below the line's largest component),
// transformed with integer additions (two instructions) and 64-bit multiplies by
// twiddles held to 63 bits, and put back to float64, by integer instructions
// throughout.  A line's scale is raised between its two radix steps only as far
// as its largest intermediate asks for, so the error of a line is a few units of
// 2^-58 .. 2^-54 of its largest component, where float64 butterflies round every
// intermediate at 2^-53 of its own size.
//
// n = 16 r (r = 4, 8, 16): a thread takes 16 points of a line, a 16-point
// transform, the twiddles, an exchange through shared memory, and 16/r r-point
// transforms.  Passes: x by pairs of real rows as one complex line (separated, or
// joined, by Hermitian symmetry), y and z in place on lines a stride apart, eight
// or more adjacent lines per block so that accesses are 128-byte segments.  Each
// pass reads and writes the array once.  Bound by the integer pipes (the 64-bit
// multiplies), at a third of the memory's rate.  Measured on GB300, one array, us,
// cuFFT -> here: 256^3 forward 1758 -> 397, inverse 1776 -> 436; 128^3 242 -> 68,
// 250 -> 79; 64^3 45 -> 36, 47 -> 39; a 32^3 array is left to cuFFT (inverse 26,
// here 36: three launches' latency).  Error against a long-double transform over
// the norm, white noise at 256^3: 2.8e-16 -> 1.0e-16; there and back 5.6e-16 ->
// 0.9e-16.
//
// A line with a value that is not finite comes out as NaN, as it would from
// float64 arithmetic after three passes.
#include "fft.h"

#include <stdint.h>

namespace pycool {

namespace {

constexpr int kFftThreads = 128;
constexpr int kTwiddles = 256;                    // of the largest n

// cos(2 pi j / 256) 2^63, j = 0 .. 64, to nearest (the first, 2^63, as 2^63 - 1)
constexpr long long kQuarterWave[kTwiddles / 4 + 1] = {
    9223372036854775807ll, 9220594129639322349ll, 9212262081300395919ll, 9198380910752360533ll,
    9178958979493303928ll, 9154007986568383775ll, 9123542961522760326ll, 9087582255348360406ll,
    9046147529429926059ll, 8999263742497006356ll, 8946959135589751977ll, 8889265215047568628ll,
    8826216733530876278ll, 8757851669087406010ll, 8684211202275644159ll, 8605339691359203716ll,
    8521284645587064995ll, 8432096696575780529ll, 8337829567810882499ll, 8238540042285863898ll,
    8134287928298226505ll, 8025136023423198846ll, 7911150076686825028ll, 7792398748961209966ll,
    7668953571605777421ll, 7540888903379453815ll, 7408281885649732303ll, 7271212395925597501ll,
    7129762999742300884ll, 6984018900926969672ll, 6834067890275007352ll, 6680000292668201229ll,
    6521908912666391106ll, 6359888978605472621ll, 6194038085235408523ll, 6024456134932800591ll,
    5851245277523433568ll, 5674509848751039730ll, 5494356307429348228ll, 5310893171315276450ll,
    5124230951741890994ll, 4934482087050512913ll, 4741760874862065242ll, 4546183403228460023ll,
    4347867480705496636ll, 4146932565389392941ll, 3943499692959694935ll, 3737691403771909211ll,
    3529631669043774883ll, 3319445816179637598ll, 3107260453277907452ll, 2893203392867074694ll,
    2677403574916221777ll, 2459990989166407361ll, 2241096596829706927ll, 2020852251703075581ll,
    1799390620744551094ll, 1576845104159639125ll, 1353349755046017570ll, 1129039198644963098ll,
    904048551248139761ll, 678513338808597222ll, 452569415305004282ll, 226352880908292031ll,
    0ll};
struct Twiddles {
  longlong2 w[kTwiddles];   // cos, sin of 2 pi j / 256, times 2^63
};
constexpr Twiddles all_twiddles() {
  Twiddles t{};
  constexpr int Q = kTwiddles / 4;
  for (int j = 0; j < kTwiddles; ++j) {
    const int r = j % Q, quad = j / Q;
    const long long c = kQuarterWave[r], s = kQuarterWave[Q - r];
    t.w[j].x = quad == 0 ? c : quad == 1 ? -s : quad == 2 ? -c : s;
    t.w[j].y = quad == 0 ? s : quad == 1 ? c : quad == 2 ? -s : -c;
  }
  return t;
}
// part of the module's image: in place before any kernel of it runs, whatever the
// stream, the thread or a capture in progress
__device__ const Twiddles g_twiddle = all_twiddles();

struct ci {
  long long re, im;
};
__device__ __forceinline__ ci operator+(ci a, ci b) { return ci{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ ci operator-(ci a, ci b) { return ci{a.re - b.re, a.im - b.im}; }
// a w, w times 2^63, rounded to nearest: a cut product is off to one side, and the
// lines of a field on a homogeneous background, nearly equal, would add that up
__device__ __forceinline__ long long mulq(long long a, long long w) {
  const __int128 p = (__int128)a * w;
  return (long long)((p + ((__int128)1 << 62)) >> 63);
}
// v (c + i DIR s)
template <int DIR> __device__ __forceinline__ ci rotate(ci v, long long c, long long s) {
  if (DIR < 0) return ci{mulq(v.re, c) + mulq(v.im, s), mulq(v.im, c) - mulq(v.re, s)};
  return ci{mulq(v.re, c) - mulq(v.im, s), mulq(v.im, c) + mulq(v.re, s)};
}
// v (DIR i)
template <int DIR> __device__ __forceinline__ ci quarter(ci v) {
  return DIR < 0 ? ci{v.im, -v.re} : ci{-v.im, v.re};
}
constexpr long long kC8 = 8521284645587064995ll;   // cos(pi/8) 2^63
constexpr long long kS8 = 3529631669043774883ll;   // sin(pi/8) 2^63
constexpr long long kR2 = 6521908912666391106ll;   // sqrt(1/2) 2^63

template <int DIR> __device__ __forceinline__ void dft4(ci& a, ci& b, ci& c, ci& d) {
  const ci t0 = a + c, t1 = a - c, t2 = b + d, t3 = quarter<DIR>(b - d);
  a = t0 + t2;
  b = t1 + t3;
  c = t0 - t2;
  d = t1 - t3;
}
// v e^(DIR i pi/4)
template <int DIR> __device__ __forceinline__ ci eighth(ci v) {
  if (DIR < 0) return ci{mulq(v.re + v.im, kR2), mulq(v.im - v.re, kR2)};
  return ci{mulq(v.re - v.im, kR2), mulq(v.im + v.re, kR2)};
}
// in place, natural order out
template <int DIR> __device__ __forceinline__ void dft8(ci (&v)[8]) {
  ci e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
  dft4<DIR>(e[0], e[1], e[2], e[3]);
  dft4<DIR>(o[0], o[1], o[2], o[3]);
  o[1] = eighth<DIR>(o[1]);
  o[2] = quarter<DIR>(o[2]);
  o[3] = eighth<DIR>(quarter<DIR>(o[3]));
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = e[k] + o[k];
    v[k + 4] = e[k] - o[k];
  }
}
template <int DIR> __device__ __forceinline__ void dft16(ci (&v)[16]) {
  // X[k1 + 4 k2] = sum_n2 w16^(n2 k1) w4^(n2 k2) sum_n1 x[4 n1 + n2] w4^(n1 k1)
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) dft4<DIR>(v[n2], v[4 + n2], v[8 + n2], v[12 + n2]);
  // now v[4 k1 + n2]
  v[4 + 1] = rotate<DIR>(v[4 + 1], kC8, kS8);
  v[4 + 2] = eighth<DIR>(v[4 + 2]);
  v[4 + 3] = rotate<DIR>(v[4 + 3], kS8, kC8);
  v[8 + 1] = eighth<DIR>(v[8 + 1]);
  v[8 + 2] = quarter<DIR>(v[8 + 2]);
  v[8 + 3] = eighth<DIR>(quarter<DIR>(v[8 + 3]));
  v[12 + 1] = rotate<DIR>(v[12 + 1], kS8, kC8);
  v[12 + 2] = eighth<DIR>(quarter<DIR>(v[12 + 2]));
  v[12 + 3] = rotate<DIR>(v[12 + 3], -kC8, -kS8);
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) dft4<DIR>(v[4 * k1], v[4 * k1 + 1], v[4 * k1 + 2], v[4 * k1 + 3]);
  // v[4 k1 + k2] = X[k1 + 4 k2]: transpose to natural order
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = i + 1; j < 4; ++j) {
      const ci t = v[4 * i + j];
      v[4 * i + j] = v[4 * j + i];
      v[4 * j + i] = t;
    }
}
// 16/R transforms of R points: point j of transform i at v[i R + j]
template <int R, int DIR> __device__ __forceinline__ void dft_rows(ci (&v)[16]) {
  if constexpr (R == 16) {
    dft16<DIR>(v);
  } else if constexpr (R == 8) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      ci w[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) w[j] = v[8 * i + j];
      dft8<DIR>(w);
#pragma unroll
      for (int j = 0; j < 8; ++j) v[8 * i + j] = w[j];
    }
  } else {
    static_assert(R == 4, "16, 8 or 4 points");
#pragma unroll
    for (int i = 0; i < 4; ++i) dft4<DIR>(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
  }
}

// v 2^(1086 - E), cut; E - (biased exponent of v) is at least 1
__device__ __forceinline__ long long to_q(double v, int E) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const int hi = __double2hiint(v);
  unsigned long long m = (b << 11) | 0x8000000000000000ull;
  asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(E - ((hi >> 20) & 0x7ff)));
  return (long long)(hi < 0 ? 0ull - m : m);
}
// x 2^(E - 1086) rounded to nearest; past the largest float64: infinity
__device__ __forceinline__ double from_q(long long x, int E) {
  const bool neg = x < 0;
  unsigned long long m = neg ? 0ull - (unsigned long long)x : (unsigned long long)x;
  const int lz = __clzll((long long)m);
  asm("shl.b64 %0, %0, %1;" : "+l"(m) : "r"(lz));
  unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);
  r += (unsigned long long)(uint32_t)(E - lz - 1) << 52;
  if (E - lz - 1 >= 2046) r = 0x7ff0000000000000ull;
  r |= neg ? 0x8000000000000000ull : 0ull;
  return __longlong_as_double((long long)(m == 0ull ? 0ull : r));
}
__device__ __forceinline__ uint32_t mag_hi(double v) {
  return (uint32_t)__double2hiint(v) & 0x7fffffffu;
}

// A line's scale from the high word of its largest component: |I| < 2^(63 - room)
template <int ROOM> __device__ __forceinline__ int line_exponent(uint32_t top) {
  return max((int)(top >> 20), 64) + ROOM + 1;
}

// The body of a pass: v holds the thread's 16 points of its line on scale E.
// 16-point step, twiddles, raise of the scale, exchange, R-point steps.  t: the
// thread's number in its line (0 .. R - 1).  s_top: the line's word for the
// maximum (zeroed before).  put(m, t, value), get(m, t): the exchange buffer.
// BITS: the largest component afterwards is below 2^(BITS + log2 R + 1/2).
template <int R, int DIR, int BITS, typename Put, typename Get>
__device__ __forceinline__ void line_transform(ci (&v)[16], int& E, int t, uint32_t* s_top,
                                               Put&& put, Get&& get) {
  dft16<DIR>(v);
  uint32_t top = 0u;
#pragma unroll
  for (int m = 0; m < 16; ++m) {
    if (m > 0) {   // w_n^(t m), 1 for the line's first thread
      const longlong2 w = g_twiddle.w[(t * m) * (kTwiddles / (16 * R))];
      const ci r = rotate<DIR>(v[m], w.x, w.y);
      v[m] = t > 0 ? r : v[m];
    }
    top = max(top, (uint32_t)((v[m].re ^ (v[m].re >> 63)) >> 32));
    top = max(top, (uint32_t)((v[m].im ^ (v[m].im >> 63)) >> 32));
  }
  atomicMax(s_top, top);
  __syncthreads();
  const int sh = max(0, 32 - __clz((int)*s_top) - (BITS - 32));
  E += sh;
  const long long half = sh > 0 ? 1ll << (sh - 1) : 0ll;
#pragma unroll
  for (int m = 0; m < 16; ++m) put(m, t, ci{(v[m].re + half) >> sh, (v[m].im + half) >> sh});
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 16 / R; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) v[i * R + j] = get(t + R * i, j);
  dft_rows<R, DIR>(v);   // v[i R + q] = X[t + R i + 16 q]
}

// Complex lines `stride` elements apart, in place: line l of slab b starts at
// data + b slab + l.
template <int R, int DIR>
__global__ void __launch_bounds__(kFftThreads) fft_lines(double2* __restrict__ data, int lines,
                                                         long long slab, long long stride) {
  constexpr int W = kFftThreads / R;   // lines per block
  __shared__ ci ex[16 * R * W];
  __shared__ uint32_t s_top[2][W];
  const int c = threadIdx.x % W, t = threadIdx.x / W;
  const int line = blockIdx.x * W + c;
  const bool valid = line < lines;
  double2* p = data + (long long)blockIdx.y * slab + line;
  if (threadIdx.x < 2 * W) s_top[threadIdx.x / W][threadIdx.x % W] = 0u;
  double2 x[16];
  uint32_t top = 0u;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    x[k] = valid ? p[(long long)(t + R * k) * stride] : make_double2(0.0, 0.0);
    top = max(top, max(mag_hi(x[k].x), mag_hi(x[k].y)));
  }
  __syncthreads();
  atomicMax(&s_top[0][c], top);
  __syncthreads();
  top = s_top[0][c];
  int E = line_exponent<5>(top);
  ci v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = ci{to_q(x[k].x, E), to_q(x[k].y, E)};
  line_transform<R, DIR, 58>(
      v, E, t, &s_top[1][c], [&](int m, int tt, ci a) { ex[(m * R + tt) * W + c] = a; },
      [&](int m, int tt) { return ex[(m * R + tt) * W + c]; });
  if (!valid) return;
  const bool bad = top >= 0x7ff00000u;
  const double nan = __hiloint2double(0x7ff80000, 0);
#pragma unroll
  for (int i = 0; i < 16 / R; ++i)
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const ci a = v[i * R + q];
      p[(long long)(t + R * i + 16 * q) * stride] =
          bad ? make_double2(nan, nan) : make_double2(from_q(a.re, E), from_q(a.im, E));
    }
}

// Pairs of real rows (n values) into half-spectrum rows (n/2 + 1): the pair is the
// complex line a + i b, Z its transform, A_k = (Z_k + conj Z_(n-k))/2 and B_k =
// (Z_k - conj Z_(n-k))/(2 i).
template <int R>
__global__ void __launch_bounds__(kFftThreads) fft_rows_real(const double* __restrict__ in,
                                                             double2* __restrict__ out) {
  constexpr int N = 16 * R, NH = N / 2 + 1, W = kFftThreads / R;
  constexpr int PAD = R + 1;   // off the banks
  __shared__ ci ex[W * 16 * PAD];
  __shared__ uint32_t s_top[2][W];
  const int c = threadIdx.x / R, t = threadIdx.x % R;
  const long long row = 2 * ((long long)blockIdx.x * W + c);   // n^2 is a multiple of 2 W
  for (int i = threadIdx.x; i < 2 * W; i += kFftThreads) s_top[i / W][i % W] = 0u;
  const double* a = in + row * N;
  double xa[16], xb[16];
  uint32_t top = 0u;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    xa[k] = __ldg(a + t + R * k);
    xb[k] = __ldg(a + N + t + R * k);
    top = max(top, max(mag_hi(xa[k]), mag_hi(xb[k])));
  }
  __syncthreads();
  atomicMax(&s_top[0][c], top);
  __syncthreads();
  top = s_top[0][c];
  int E = line_exponent<5>(top);
  ci v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = ci{to_q(xa[k], E), to_q(xb[k], E)};
  ci* const line = ex + c * 16 * PAD;
  line_transform<R, -1, 57>(
      v, E, t, &s_top[1][c], [&](int m, int tt, ci z) { line[m * PAD + tt] = z; },
      [&](int m, int tt) { return line[m * PAD + tt]; });
  __syncthreads();   // every thread has read its points
#pragma unroll
  for (int i = 0; i < 16 / R; ++i)
#pragma unroll
    for (int q = 0; q < R; ++q) line[t + R * i + 16 * q] = v[i * R + q];
  __syncthreads();
  const bool bad = top >= 0x7ff00000u;
  const double nan = __hiloint2double(0x7ff80000, 0);
  double2* oa = out + row * NH;
  for (int k = t; k <= N / 2; k += R) {
    const ci z = line[k], y = line[k == 0 ? 0 : N - k];
    double2 A = make_double2(from_q(z.re + y.re, E - 1), from_q(z.im - y.im, E - 1));
    double2 B = make_double2(from_q(z.im + y.im, E - 1), from_q(y.re - z.re, E - 1));
    if (bad) A = B = make_double2(nan, nan);
    oa[k] = A;
    oa[NH + k] = B;
  }
}

// The inverse: Z_k = A_k + i B_k, Z_(n-k) = conj A_k + i conj B_k; the imaginary
// parts of A and B at k = 0 and n/2 do not count.
template <int R>
__global__ void __launch_bounds__(kFftThreads) fft_rows_real_inv(const double2* __restrict__ in,
                                                                 double* __restrict__ out) {
  constexpr int N = 16 * R, NH = N / 2 + 1, W = kFftThreads / R;
  constexpr int PAD = R + 1;   // off the banks
  __shared__ ci ex[W * 16 * PAD];
  __shared__ uint32_t s_top[2][W];
  const int c = threadIdx.x / R, t = threadIdx.x % R;
  const long long row = 2 * ((long long)blockIdx.x * W + c);
  for (int i = threadIdx.x; i < 2 * W; i += kFftThreads) s_top[i / W][i % W] = 0u;
  const double2* a = in + row * NH;
  uint32_t top = 0u;
  for (int k = t; k < NH; k += R) {
    const double2 A = a[k], B = a[NH + k];
    top = max(top, max(max(mag_hi(A.x), mag_hi(A.y)), max(mag_hi(B.x), mag_hi(B.y))));
  }
  __syncthreads();
  atomicMax(&s_top[0][c], top);
  __syncthreads();
  top = s_top[0][c];
  int E = line_exponent<6>(top);
  ci v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int j = t + R * k, jj = j <= N / 2 ? j : N - j;
    const double2 A = a[jj], B = a[NH + jj];
    const bool real = jj == 0 || jj == N / 2;
    const long long ar = to_q(A.x, E), br = to_q(B.x, E);
    const long long ai = real ? 0ll : to_q(A.y, E), bi = real ? 0ll : to_q(B.y, E);
    v[k] = j <= N / 2 ? ci{ar - bi, ai + br} : ci{ar + bi, br - ai};
  }
  ci* const line = ex + c * 16 * PAD;
  line_transform<R, 1, 58>(
      v, E, t, &s_top[1][c], [&](int m, int tt, ci z) { line[m * PAD + tt] = z; },
      [&](int m, int tt) { return line[m * PAD + tt]; });
  const bool bad = top >= 0x7ff00000u;
  const double nan = __hiloint2double(0x7ff80000, 0);
  double* oa = out + row * N;
#pragma unroll
  for (int i = 0; i < 16 / R; ++i)
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const ci z = v[i * R + q];
      const int x = t + R * i + 16 * q;
      oa[x] = bad ? nan : from_q(z.re, E);
      oa[N + x] = bad ? nan : from_q(z.im, E);
    }
}

template <int R> cudaError_t forward(const double* in, double2* out, int batch, cudaStream_t s) {
  constexpr int N = 16 * R, NH = N / 2 + 1, W = kFftThreads / R;
  constexpr long long half = (long long)N * N * NH;
  fft_rows_real<R><<<(unsigned)((long long)batch * N * N / (2 * W)), kFftThreads, 0, s>>>(in, out);
  fft_lines<R, -1><<<dim3((NH + W - 1) / W, batch * N), kFftThreads, 0, s>>>(out, NH,
                                                                            (long long)N * NH, NH);
  fft_lines<R, -1><<<dim3((N * NH + W - 1) / W, batch), kFftThreads, 0, s>>>(
      out, N * NH, half, (long long)N * NH);
  return cudaGetLastError();
}
template <int R> cudaError_t inverse(double2* spec, double* out, int batch, cudaStream_t s) {
  constexpr int N = 16 * R, NH = N / 2 + 1, W = kFftThreads / R;
  constexpr long long half = (long long)N * N * NH;
  fft_lines<R, 1><<<dim3((N * NH + W - 1) / W, batch), kFftThreads, 0, s>>>(
      spec, N * NH, half, (long long)N * NH);
  fft_lines<R, 1><<<dim3((NH + W - 1) / W, batch * N), kFftThreads, 0, s>>>(spec, NH,
                                                                           (long long)N * NH, NH);
  fft_rows_real_inv<R><<<(unsigned)((long long)batch * N * N / (2 * W)), kFftThreads, 0, s>>>(spec,
                                                                                             out);
  return cudaGetLastError();
}

}  // namespace

cudaError_t fft_forward(const double* in, double2* out, int n, int batch, cudaStream_t s) {
  switch (n) {
    case 64: return forward<4>(in, out, batch, s);
    case 128: return forward<8>(in, out, batch, s);
    case 256: return forward<16>(in, out, batch, s);
  }
  return cudaErrorInvalidValue;
}
cudaError_t fft_inverse(double2* spec, double* out, int n, int batch, cudaStream_t s) {
  switch (n) {
    case 64: return inverse<4>(spec, out, batch, s);
    case 128: return inverse<8>(spec, out, batch, s);
    case 256: return inverse<16>(spec, out, batch, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace pycool
