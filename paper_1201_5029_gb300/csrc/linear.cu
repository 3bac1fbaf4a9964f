// Growth functions of the linearised evolution (Sec. 2.2): the background
// fields, a and p_a evolve without the perturbations (H^(2) neglected, Eqs.
// a-lin, phi-0) and every Fourier mode of the perturbations obeys the linear
// equations of Eq. Phik-1, in which a mode enters only through k_eff^2.  One
// thread takes one distinct k_eff^2 and advances the 2N_f x 2N_f transfer
// matrix T of its modes, (dPhi, dPi)(eta) = T (dPhi, dPi)(0), through the same
// split-Hamiltonian stages as the lattice (Sec. 2.3):
//   Phi_H1(h): a   -= p_a h / (6 V_L m_pl^2)
//   Phi_H2(h): p_a += V_L [sum_i pi0_i^2 / a^3 - rho_m0] h,
//              phi0 += pi0 h / a^2,   T_dPhi += T_dPi h / a^2
//   Phi_H3(h): p_a -= 4 V_L a^3 V(phi0) h,   pi0 -= a^4 V'(phi0) h,
//              T_dPi -= [k_eff^2 a^2 / dx^2 + a^4 M(phi0)] T_dPhi h
// with M the matrix of second derivatives of V at the background.
//
// The background and with it the coefficients of every stage are the same for
// all modes, so one thread walks the chain of stages (a division and some
// twenty dependent float64 operations each) and writes the coefficients to a
// table, and the threads of the k_eff^2 values only apply them: 26 float64
// instructions per stage for two fields, where a thread that evolved its own
// background spent about 350.  The walk runs one chunk of stages ahead of the
// modes, in the same launches.  Bound by the float64 pipe.  Measured on GB300,
// 128^3 two-field lattice, 300 stages: the growth functions 8.5 -> 1.09 ms (a
// chunk of 64 stages: 0.15 ms for the walk alone, 0.15 for the modes alone, 0.22
// together, since the walk shares one scheduler's float64 pipe).
#include <cufft.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <tuple>
#include <vector>

#include "internal.cuh"
#include "fft.h"
#include "models.cuh"
#include "runtime.h"

namespace pycool {

constexpr int kLinChunk = 64;   // stages per launch
struct LinEntry {               // one stage for the modes: T_dPhi += c T_dPi, then
  double c, kq, M[3];           //   T_dPi -= (q kq + M) T_dPhi,  M = M00, M01, M11 (times a^4 h)
};
struct LinState {               // the background between launches
  double A, PA, f0[2], p0[2], deta, cprev;   // cprev: the last stage's trailing drift
};

struct LinArgs {
  const double* k2;       // k_eff^2 values (dimensionless symbols)
  long long nk;
  double* T;              // out: nk x (2N_f)^2, row-major (rows dPhi_0.., dPi_0..)
  double* bg;             // out: a, p_a, phi0[N_f], pi0[N_f]
  LinEntry* table;        // [2][kLinChunk]
  LinState* state;
  long long chunk, nentries;   // this launch's chunk; stages + 1 (the last trailing drift)
  const double* bg_in;    // device: initial phi0[N_f], pi0[N_f] (NULL: the fields below)
  double a0, pa0, phi0[2], pi0[2];
  double w[kMaxStages];
  int nstages;
  long long steps;
  int physical;           // d-eta = dt / a at each step's start (Sec. 3.1), else dt
  double dt, dx2inv, VL, inv6VLm2, rho_m0;
  double params[8], derived[4];
};

// Second derivatives of the potentials of Sec. 3 at the background.
template <int MODEL> struct Hess;
template <> struct Hess<M_FREE> {
  __device__ static void get(const double* p, const double*, const double*, double (&M)[1][1]) {
    M[0][0] = p[0];
  }
};
template <> struct Hess<M_CHAOTIC2> {   // V = m2 phi^2/2 + g2 phi^2 chi^2/2
  __device__ static void get(const double* p, const double*, const double* f, double (&M)[2][2]) {
    M[0][0] = p[0] + p[1] * f[1] * f[1];
    M[0][1] = M[1][0] = 2.0 * p[1] * f[0] * f[1];
    M[1][1] = p[1] * f[0] * f[0];
  }
};
template <> struct Hess<M_OSCILLON> {   // V = m2 x^2/2 - lam x^4/4 + g x^6/6
  __device__ static void get(const double* p, const double*, const double* f, double (&M)[1][1]) {
    const double x2 = f[0] * f[0];
    M[0][0] = p[0] - 3.0 * p[1] * x2 + 5.0 * p[2] * x2 * x2;
  }
};
template <> struct Hess<M_QBALL> {      // V = m2 u (1 + K ln(u/M^2)), u = |phi|^2/2
  __device__ static void get(const double* p, const double* dv, const double* f,
                             double (&M)[2][2]) {
    const double u = 0.5 * (f[0] * f[0] + f[1] * f[1]);
    const double fac = p[0] * (1.0 + p[1] + p[1] * (log(u) - dv[0]));
    const double c = p[0] * p[1] / u;
    M[0][0] = fac + c * f[0] * f[0];
    M[0][1] = M[1][0] = c * f[0] * f[1];
    M[1][1] = fac + c * f[1] * f[1];
  }
};

// The background through the entries [e0, e1) of the table (one thread).  An
// entry is the drift that two stages share, then the later one's kick; the last
// entry is the last stage's trailing drift alone.
template <int MODEL>
__device__ void linear_background(const LinArgs& a, LinEntry* out, long long e0, long long e1) {
  using P = Pot<MODEL>;
  constexpr int NF = P::NF;
  const typename P::K pk = P::prep(a.params, a.derived);
  LinState b;
  if (e0 == 0) {
    b.A = a.a0;
    b.PA = a.pa0;
    b.deta = a.dt;
    b.cprev = 0.0;
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      b.f0[i] = a.bg_in ? a.bg_in[i] : a.phi0[i];
      b.p0[i] = a.bg_in ? a.bg_in[NF + i] : a.pi0[i];
    }
  } else {
    b = *a.state;
  }
  int stage = (int)(e0 % a.nstages);
  for (long long e = e0; e < e1; ++e) {
    LinEntry t;
    if (e == a.nentries - 1) {
      t.c = b.cprev;
      t.kq = t.M[0] = t.M[1] = t.M[2] = 0.0;
      out[e - e0] = t;
      break;
    }
    if (stage == 0 && a.physical) b.deta = a.dt / b.A;   // the step's start
    const double h = a.w[stage] * b.deta, hh = 0.5 * h;
    b.A = b.A - b.PA * a.inv6VLm2 * hh;
    const double ia = 1.0 / b.A, ia2 = ia * ia, a2 = b.A * b.A, a4 = a2 * a2;
    const double c = hh * ia2;
    auto h2 = [&]() {   // Phi_H2(h/2): p_a and the background fields
      double s2 = 0.0;
#pragma unroll
      for (int i = 0; i < NF; ++i) s2 += b.p0[i] * b.p0[i];
      b.PA = b.PA + a.VL * (s2 * (ia2 * ia) - a.rho_m0) * hh;
#pragma unroll
      for (int i = 0; i < NF; ++i) b.f0[i] = b.f0[i] + b.p0[i] * c;
    };
    h2();
    double dV[NF], V, M[NF][NF];
    P::eval(pk, b.f0, dV, V);
    Hess<MODEL>::get(a.params, a.derived, b.f0, M);
    t.c = b.cprev + c;
    t.kq = a2 * h;
    const double a4h = a4 * h;
    t.M[0] = a4h * M[0][0];
    t.M[1] = NF > 1 ? a4h * M[0][NF - 1] : 0.0;
    t.M[2] = NF > 1 ? a4h * M[NF - 1][NF - 1] : 0.0;
    out[e - e0] = t;
    b.PA = b.PA - 4.0 * a.VL * (a2 * b.A) * V * h;
#pragma unroll
    for (int i = 0; i < NF; ++i) b.p0[i] = b.p0[i] - a4h * dV[i];
    h2();
    b.A = b.A - b.PA * a.inv6VLm2 * hh;
    b.cprev = c;
    if (++stage == a.nstages) stage = 0;
  }
  *a.state = b;
  if (e1 == a.nentries) {
    a.bg[0] = b.A;
    a.bg[1] = b.PA;
#pragma unroll
    for (int i = 0; i < NF; ++i) { a.bg[2 + i] = b.f0[i]; a.bg[2 + NF + i] = b.p0[i]; }
  }
}

// Launch `chunk`: block 0 forms that chunk's table, the others apply the chunk
// before it to the transfer matrices.  Block 0's one thread is a chain of float64
// instructions that waits for the pipe behind every other warp of its scheduler.
// With 64 values a block, more blocks than SMs put two or three warps there.  Where
// all values fit one wave of two blocks of five warps to an SM (by their shared
// memory), block 0 has one other block beside it instead: 128^3 (48 000 values), a
// chunk 220 -> 181 us, the whole linearised evolution of 300 stages 2123 -> 2009 us.
// Fewer values have the SM to themselves, and several waves gain nothing (256^3
// 7.64 -> 7.76 ms).
constexpr int kLinThreads = 160;
constexpr int kLinSmem = 96 * 1024;   // of an SM's 228 KB: two blocks fit, three do not
template <int MODEL>
__global__ void __launch_bounds__(kLinThreads) linear_growth(const LinArgs a) {
  constexpr int NF = Pot<MODEL>::NF, N2 = 2 * NF;
  __shared__ LinEntry tab[kLinChunk];
  if (blockIdx.x == 0) {
    const long long e0 = a.chunk * kLinChunk;
    if (threadIdx.x == 0 && e0 < a.nentries)
      linear_background<MODEL>(a, a.table + (a.chunk & 1) * kLinChunk, e0,
                               min(e0 + kLinChunk, a.nentries));
    return;
  }
  const long long e0 = (a.chunk - 1) * kLinChunk;
  const int ne = (int)min((long long)kLinChunk, a.nentries - e0);
  const LinEntry* src = a.table + ((a.chunk - 1) & 1) * kLinChunk;
  for (int i = threadIdx.x; i < ne; i += blockDim.x) tab[i] = src[i];
  __syncthreads();
  const long long k = (long long)(blockIdx.x - 1) * blockDim.x + threadIdx.x;
  if (k >= a.nk) return;
  const double q = a.k2[k] * a.dx2inv;   // k_eff^2 / dx^2
  double* out = a.T + (size_t)k * N2 * N2;
  double T[N2][N2];
#pragma unroll
  for (int r = 0; r < N2; ++r)
#pragma unroll
    for (int c = 0; c < N2; ++c) T[r][c] = e0 > 0 ? out[r * N2 + c] : ((r == c) ? 1.0 : 0.0);
  for (int e = 0; e < ne; ++e) {
    const LinEntry t = tab[e];
#pragma unroll
    for (int i = 0; i < NF; ++i)
#pragma unroll
      for (int c = 0; c < N2; ++c) T[i][c] = fma(t.c, T[NF + i][c], T[i][c]);
    const double k00 = fma(q, t.kq, t.M[0]), k11 = fma(q, t.kq, t.M[2]);
#pragma unroll
    for (int c = 0; c < N2; ++c) {
      if constexpr (NF == 1) {
        T[1][c] = fma(-k00, T[0][c], T[1][c]);
      } else {
        T[2][c] = fma(-k00, T[0][c], fma(-t.M[1], T[1][c], T[2][c]));
        T[3][c] = fma(-k11, T[1][c], fma(-t.M[1], T[0][c], T[3][c]));
      }
    }
  }
#pragma unroll
  for (int r = 0; r < N2; ++r)
#pragma unroll
    for (int c = 0; c < N2; ++c) out[r * N2 + c] = T[r][c];
}

// Scratch of launch_linear_growth, after the caller's background slots.
constexpr size_t kLinScratch = 2 * kLinChunk * sizeof(LinEntry) + sizeof(LinState);

cudaError_t launch_linear_growth(int model, LinArgs a, void* scratch, cudaStream_t s) {
  a.table = static_cast<LinEntry*>(scratch);
  a.state = reinterpret_cast<LinState*>(a.table + 2 * kLinChunk);
  a.nentries = a.steps * a.nstages + 1;
  const long long chunks = (a.nentries + kLinChunk - 1) / kLinChunk;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const bool wide = (a.nk + 63) / 64 > sms && (a.nk + kLinThreads - 1) / kLinThreads < 2ll * sms;
  const int threads = wide ? kLinThreads : 64, smem = wide ? kLinSmem : 0;
  auto run = [&](auto* kernel) -> cudaError_t {
    if (wide) {
      const cudaError_t ae = cudaFuncSetAttribute(
          kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kLinSmem);
      if (ae != cudaSuccess) return ae;
    }
    for (a.chunk = 0; a.chunk <= chunks; ++a.chunk) {
      const unsigned grid =
          1 + (a.chunk > 0 ? (unsigned)((a.nk + threads - 1) / threads) : 0u);
      kernel<<<grid, threads, smem, s>>>(a);
      const cudaError_t le = cudaGetLastError();
      if (le != cudaSuccess) return le;
    }
    return cudaSuccess;
  };
  switch (model) {
    case M_FREE: return run(linear_growth<M_FREE>);
    case M_CHAOTIC2: return run(linear_growth<M_CHAOTIC2>);
    case M_OSCILLON: return run(linear_growth<M_OSCILLON>);
    case M_QBALL: return run(linear_growth<M_QBALL>);
    default: return cudaErrorInvalidValue;
  }
}

// The modes of an n^3 lattice by the magnitudes of their wave numbers: k_eff^2
// is even and symmetric in them, so the modes whose sorted magnitudes i >= j >=
// k (0 .. n/2) agree share one value, class i (i+1)(i+2)/6 + j (j+1)/2 + k.  A
// mode's class is a few integer instructions, where a table of classes would
// have to be made on the host and copied (4.3 MB for 128^3).  A few classes
// hold equal values (47 905 classes, 45 760 values for 128^3).
__host__ __device__ __forceinline__ long long linear_class(int i, int j, int k) {
  const int hi = max(i, max(j, k)), lo = min(i, min(j, k)), mid = i + j + k - hi - lo;
  return (long long)hi * (hi + 1) * (hi + 2) / 6 + (long long)mid * (mid + 1) / 2 + lo;
}
struct LinSymbol {       // cos(2 pi m / n), m = 0 .. n/2, and the 13-point axis part
  double cs[257], ax4[257];
};
__global__ void __launch_bounds__(256) linear_k2(const __grid_constant__ LinSymbol sy, int half_n,
                                                 int stencil, double* k2) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y, i = blockIdx.z;
  if (k > j || j > i || i > half_n) return;
  const double cz = sy.cs[i], cy = sy.cs[j], cx = sy.cs[k];
  double v;
  if (stencil == PYCOOL_STENCIL_4TH)
    v = 90.0 / 12.0 + sy.ax4[i] + sy.ax4[j] + sy.ax4[k];
  else if (stencil == PYCOOL_STENCIL_7PT)
    v = 6.0 - 2.0 * (cz + cy + cx);
  else
    v = 128.0 / 30.0 - (2.0 * (14.0 / 30.0) * (cz + cy + cx) +
                        4.0 * (3.0 / 30.0) * (cz * cy + cz * cx + cy * cx) +
                        8.0 * (1.0 / 30.0) * cz * cy * cx);
  k2[linear_class(i, j, k)] = v;
}

// The background of lattice fields (Eq. phi-lin): the lattice means of the
// 2 N_f arrays phi_0..phi_{N-1}, pi_0.. (src[j] = array j, S values each),
// summed in a fixed order -- per block a strided range and a fixed tree, then
// the block sums in order by one block -- so the means are reproducible.
constexpr int kMeanBlocks = 128;
__global__ void __launch_bounds__(256) linear_means_partial(const double* const* src, long long S,
                                                            double* part) {
  __shared__ double red[256];
  const int j = blockIdx.y;
  double acc = 0.0;
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < S; i += (long long)kMeanBlocks * 256)
    acc += src[j][i];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[(size_t)j * kMeanBlocks + blockIdx.x] = red[0];
}
__global__ void linear_means_fold(const double* part, int narr, double invS, double* bg_in) {
  const int j = threadIdx.x;   // one thread per array
  if (j >= narr) return;
  double s = 0.0;
  for (int b = 0; b < kMeanBlocks; ++b) s += part[(size_t)j * kMeanBlocks + b];
  bg_in[j] = s * invS;         // [phi0_0 .. phi0_{N_f-1}, pi0_0 ..]
}
// dst_f = src_f - mean_f (the perturbations, Eq. phi-lin), into the output
// arrays that later receive the evolved fields
__global__ void linear_subtract(const double* const* src, double* const* dst, long long S,
                                int narr, const double* bg_in) {
  const long long total = S * narr;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int j = (int)(i / S);
    const long long e = i - (long long)j * S;
    dst[j][e] = src[j][e] - bg_in[j];
  }
}
// the k = 0 coefficients of the perturbations (zero up to rounding) cleared
__global__ void linear_clear_mean(cufftDoubleComplex* spec, long long half, int nf) {
  const int i = threadIdx.x;
  if (i >= 2 * nf) return;
  spec[(size_t)i * half].x = 0.0;
  spec[(size_t)i * half].y = 0.0;
}

// Each Fourier mode of the perturbations at the later time from its initial
// value (Sec. 2.2, after Eq. Phik-1): y(eta) = T[k_eff^2 of the mode] y(0),
// y = (dPhi_1..dPhi_N, dPi_1..dPi_N), T real, scaled by 1/S for the
// unnormalised inverse transform; the k = 0 coefficient becomes the evolved
// background, so the inverse transform gives background + perturbations.
template <int NF>
__global__ void __launch_bounds__(256) linear_apply(cufftDoubleComplex* __restrict__ spec,
                                                    long long half,
                                                    int n, const double* __restrict__ T,
                                                    const double* __restrict__ bg_end, double invS) {
  constexpr int N2 = 2 * NF;
  for (long long m = blockIdx.x * (long long)blockDim.x + threadIdx.x; m < half;
       m += (long long)gridDim.x * blockDim.x) {
    cufftDoubleComplex y[N2], r[N2];
#pragma unroll
    for (int j = 0; j < N2; ++j) y[j] = spec[(size_t)j * half + m];
    if (m == 0) {
#pragma unroll
      for (int j = 0; j < N2; ++j) { r[j].x = bg_end[2 + j]; r[j].y = 0.0; }
    } else {
      const unsigned nh = n / 2 + 1, row = (unsigned)(m / nh);
      const int mx = (int)(m - (long long)row * nh), my = (int)(row % (unsigned)n),
                mz = (int)(row / (unsigned)n);
      const double* t = T + (size_t)linear_class(mx, min(my, n - my), min(mz, n - mz)) * N2 * N2;
#pragma unroll
      for (int i = 0; i < N2; ++i) {
        double re = 0.0, im = 0.0;
#pragma unroll
        for (int j = 0; j < N2; ++j) {
          const double tij = __ldg(&t[i * N2 + j]);
          re = fma(tij, y[j].x, re);
          im = fma(tij, y[j].y, im);
        }
        r[i].x = re * invS;
        r[i].y = im * invS;
      }
    }
#pragma unroll
    for (int j = 0; j < N2; ++j) spec[(size_t)j * half + m] = r[j];
  }
}

cudaError_t launch_linear_apply(int nf, cufftDoubleComplex* spec, long long half,
                                int n, const double* T, const double* bg_end, double invS,
                                cudaStream_t s) {
  const long long want = (half + 255) / 256;
  const unsigned grid = (unsigned)std::min<long long>(want, 152LL * 16);
  if (nf == 1)
    linear_apply<1><<<grid, 256, 0, s>>>(spec, half, n, T, bg_end, invS);
  else
    linear_apply<2><<<grid, 256, 0, s>>>(spec, half, n, T, bg_end, invS);
  return cudaGetLastError();
}

// The distinct k_eff^2 values (ascending) of an n^3 lattice and each mode's
// index into them (modes in numpy FFT order, [z][y][x]).
bool linear_modes_host(int n, int stencil, std::vector<double>& vals, std::vector<int32_t>* index) {
  // coefficients by neighbour class (number of non-zero offsets), Eq. D
  const double c7[4] = {-6.0, 1.0, 0.0, 0.0};
  const double c27[4] = {-128.0 / 30.0, 14.0 / 30.0, 3.0 / 30.0, 1.0 / 30.0};
  const double* c = stencil == PYCOOL_STENCIL_7PT ? c7 : c27;
  const bool fourth = stencil == PYCOOL_STENCIL_4TH;
  // one axis: wave number m (numpy FFT order) -> cos(2 pi m / n); the
  // fourth-order stencil's part of one axis, -(2 (16/12) cos t - 2 (1/12) cos 2t)
  std::vector<double> cs(n), ax4(n);
  for (int m = 0; m < n; ++m) {
    const int mm = m <= (n - 1) / 2 ? m : m - n;
    cs[m] = std::cos(2.0 * M_PI * mm / n);
    ax4[m] = -(2.0 * (16.0 / 12.0) * cs[m] + 2.0 * (-1.0 / 12.0) * std::cos(4.0 * M_PI * mm / n));
  }
  const size_t S = (size_t)n * n * n;
  std::vector<double> k2(S);
  for (int z = 0; z < n; ++z)
    for (int y = 0; y < n; ++y)
      for (int x = 0; x < n; ++x) {
        const double cz = cs[z], cy = cs[y], cx = cs[x];
        double v;
        if (fourth) {   // the centre (-90/12) and the two sites each way along every axis
          v = 90.0 / 12.0 + ax4[z] + ax4[y] + ax4[x];
        } else {
          // sum over the offsets of each class of c_d cos(k.o): products of cosines
          const double sym = c[0] + 2.0 * c[1] * (cz + cy + cx) +
                             4.0 * c[2] * (cz * cy + cz * cx + cy * cx) +
                             8.0 * c[3] * cz * cy * cx;
          v = -sym;
        }
        k2[((size_t)z * n + y) * n + x] = v;
      }
  std::vector<double> sorted(k2);
  std::sort(sorted.begin(), sorted.end());
  vals.clear();
  for (double v : sorted)
    if (vals.empty() || v - vals.back() > 1e-12 * std::fmax(1.0, std::fabs(v))) vals.push_back(v);
  if (index) {
    index->resize(S);
    for (size_t i = 0; i < S; ++i) {
      // the last value not above k2[i] + tolerance
      const double v = k2[i];
      auto it = std::upper_bound(vals.begin(), vals.end(), v + 1e-12 * std::fmax(1.0, std::fabs(v)));
      (*index)[i] = (int32_t)((it - vals.begin()) - 1);
    }
  }
  return true;
}

// Per-process cache of pycool_linear_evolve: the forward/inverse FFT plans per
// (n, N_f, device).  A plan is used under its own lock (its stream is set per
// call).
struct LinPlans {
  cufftHandle fwd = 0, inv = 0;
  std::mutex mu;
};
std::mutex g_lin_mu;
std::map<std::tuple<int, int, int>, std::shared_ptr<LinPlans>> g_lin_plans;

std::shared_ptr<LinPlans> linear_plans(int n, int nf, int device) {
  std::lock_guard<std::mutex> lk(g_lin_mu);
  auto key = std::make_tuple(n, nf, device);
  auto it = g_lin_plans.find(key);
  if (it != g_lin_plans.end()) return it->second;
  auto p = std::make_shared<LinPlans>();
  int dims[3] = {n, n, n};
  const int S = n * n * n, half = n * n * (n / 2 + 1);
  if (cufftPlanMany(&p->fwd, 3, dims, nullptr, 1, S, nullptr, 1, half, CUFFT_D2Z, nf) !=
      CUFFT_SUCCESS)
    return nullptr;
  if (cufftPlanMany(&p->inv, 3, dims, nullptr, 1, half, nullptr, 1, S, CUFFT_Z2D, nf) !=
      CUFFT_SUCCESS) {
    cufftDestroy(p->fwd);
    return nullptr;
  }
  g_lin_plans.emplace(key, p);
  return p;
}

}  // namespace pycool

using namespace pycool;

// The distinct values of k_eff^2 (the symbol of -D on plane waves, Eq. D)
// over the n^3 lattice modes, and each mode's index into them.  Values that
// differ by less than 1e-12 (equal symbols reached through different cosines)
// count as one.
extern "C" __attribute__((visibility("default"))) pycool_status pycool_linear_modes(
    int32_t n, int32_t stencil, double* values, int64_t cap, int64_t* count, int32_t* index) {
  if (n < 1 || n > 512 || !count || cap < 0 ||
      (stencil != PYCOOL_STENCIL_7PT && stencil != PYCOOL_STENCIL_ISO27 &&
       stencil != PYCOOL_STENCIL_4TH))
    return PYCOOL_E_INVALID;
  std::vector<double> vals;
  std::vector<int32_t> idx;
  linear_modes_host(n, stencil, vals, index ? &idx : nullptr);
  *count = (int64_t)vals.size();
  if (values) {
    if (cap < (int64_t)vals.size()) return PYCOOL_E_INVALID;
    for (size_t i = 0; i < vals.size(); ++i) values[i] = vals[i];
  }
  if (index) std::memcpy(index, idx.data(), idx.size() * sizeof(int32_t));
  return PYCOOL_OK;
}

extern "C" __attribute__((visibility("default"))) pycool_status pycool_linear_growth(
    const pycool_config* cfg, double a0, double pa0, const double* phi0, const double* pi0,
    const double* k2, int64_t nk, int64_t steps, double* T, double* background,
    void* cuda_stream) {
  const pycool_status v = validate(cfg);
  if (v != PYCOOL_OK) return v;
  if (cfg->model >= kRuntimeModelBase) return PYCOOL_E_INVALID;   // no second derivatives
  if (!phi0 || !pi0 || !k2 || !T || !background || nk < 1 || steps < 0 || !(a0 > 0.0) ||
      !std::isfinite(pa0))
    return PYCOOL_E_INVALID;
  const int nf = model_nfields(cfg->model);
  LinArgs a;
  std::memset(&a, 0, sizeof(a));
  a.nk = nk;
  a.a0 = a0;
  a.pa0 = pa0;
  for (int i = 0; i < nf; ++i) { a.phi0[i] = phi0[i]; a.pi0[i] = pi0[i]; }
  a.nstages = stage_table(cfg->order, a.w);
  a.steps = steps;
  a.dt = cfg->dt;
  a.physical = cfg->time_step == PYCOOL_TIME_PHYSICAL ? 1 : 0;
  const double dx = cfg->L / cfg->n;
  a.dx2inv = 1.0 / (dx * dx);
  a.VL = (double)cfg->n * cfg->n * cfg->n;
  a.inv6VLm2 = std::isinf(cfg->mpl) ? 0.0 : 1.0 / (6.0 * a.VL * cfg->mpl * cfg->mpl);
  a.rho_m0 = cfg->rho_mat0;
  for (int i = 0; i < 8; ++i) a.params[i] = cfg->params[i];
  if (cfg->model == PYCOOL_MODEL_QBALL) a.derived[0] = std::log(cfg->params[2] * cfg->params[2]);
  const size_t n2 = (size_t)(2 * nf) * (2 * nf);
  cudaStream_t s = (cudaStream_t)cuda_stream;
  double *dk = nullptr, *dT = nullptr, *dbg = nullptr;
  pycool_status st = PYCOOL_OK;
  if (cudaMalloc((void**)&dk, (size_t)nk * sizeof(double)) != cudaSuccess ||
      cudaMalloc((void**)&dT, (size_t)nk * n2 * sizeof(double)) != cudaSuccess ||
      cudaMalloc((void**)&dbg, 16 * sizeof(double) + kLinScratch) != cudaSuccess) {
    st = PYCOOL_E_NOMEM;
  } else {
    a.k2 = dk;
    a.T = dT;
    a.bg = dbg;
    if (cudaMemcpyAsync(dk, k2, (size_t)nk * sizeof(double), cudaMemcpyHostToDevice, s) !=
            cudaSuccess ||
        launch_linear_growth(cfg->model, a, dbg + 16, s) != cudaSuccess ||
        cudaMemcpyAsync(T, dT, (size_t)nk * n2 * sizeof(double), cudaMemcpyDeviceToHost, s) !=
            cudaSuccess ||
        cudaMemcpyAsync(background, dbg, (size_t)(2 + 2 * nf) * sizeof(double),
                        cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
      st = PYCOOL_E_CUDA;
  }
  cudaFree(dk);
  cudaFree(dT);
  cudaFree(dbg);
  return st;
}

// The whole linearised evolution of lattice fields on the device.
extern "C" __attribute__((visibility("default"))) pycool_status pycool_linear_evolve(
    const pycool_config* cfg, double a0, double pa0, const double* phi, const double* pi,
    int64_t steps, double* phi_out, double* pi_out, double* background, void* cuda_stream) {
  const pycool_status v = validate(cfg);
  if (v != PYCOOL_OK) return v;
  if (cfg->model >= kRuntimeModelBase) return PYCOOL_E_INVALID;   // no second derivatives
  if (!phi || !pi || !phi_out || !pi_out || !background || steps < 0 || !(a0 > 0.0) ||
      !std::isfinite(pa0) || cfg->n < 2 || cfg->n > 512)
    return PYCOOL_E_INVALID;
  {  // the outputs serve as scratch while the inputs are read: no overlap
    const size_t bytes = (size_t)model_nfields(cfg->model) * cfg->n * cfg->n * cfg->n * 8;
    const uintptr_t in[2] = {(uintptr_t)phi, (uintptr_t)pi};
    const uintptr_t out[2] = {(uintptr_t)phi_out, (uintptr_t)pi_out};
    for (int i = 0; i < 2; ++i)
      for (int j = 0; j < 2; ++j)
        if (out[i] < in[j] + bytes && in[j] < out[i] + bytes) return PYCOOL_E_INVALID;
    if (out[0] < out[1] + bytes && out[1] < out[0] + bytes) return PYCOOL_E_INVALID;
  }
  const int nf = model_nfields(cfg->model);
  const int n = cfg->n;
  const long long S = (long long)n * n * n;
  const long long half = (long long)n * n * (n / 2 + 1);   // coefficients of a real transform
  int device = 0;
  if (cudaGetDevice(&device) != cudaSuccess) return PYCOOL_E_CUDA;
  // the library's own transforms where they take the side, else cuFFT's plans
  const bool own_fft = fft_takes(n);
  std::shared_ptr<LinPlans> plans;
  std::unique_lock<std::mutex> plan_lock;
  if (!own_fft) {
    plans = linear_plans(n, nf, device);
    if (!plans) return PYCOOL_E_CUDA;
    plan_lock = std::unique_lock<std::mutex>(plans->mu);
  }
  const int hn = n / 2;
  const long long nk = linear_class(hn, hn, hn) + 1;
  const size_t N2 = (size_t)(2 * nf) * (2 * nf);

  LinArgs a;
  std::memset(&a, 0, sizeof(a));
  a.nk = nk;
  a.a0 = a0;
  a.pa0 = pa0;
  a.nstages = stage_table(cfg->order, a.w);
  a.steps = steps;
  a.dt = cfg->dt;
  a.physical = cfg->time_step == PYCOOL_TIME_PHYSICAL ? 1 : 0;
  const double dx = cfg->L / n;
  a.dx2inv = 1.0 / (dx * dx);
  a.VL = (double)S;
  a.inv6VLm2 = std::isinf(cfg->mpl) ? 0.0 : 1.0 / (6.0 * a.VL * cfg->mpl * cfg->mpl);
  a.rho_m0 = cfg->rho_mat0;
  for (int i = 0; i < 8; ++i) a.params[i] = cfg->params[i];
  if (cfg->model == PYCOOL_MODEL_QBALL) a.derived[0] = std::log(cfg->params[2] * cfg->params[2]);

  cudaStream_t s = (cudaStream_t)cuda_stream;
  cufftDoubleComplex* spec = nullptr;   // [phi, pi][N_f][half]
  double *dk = nullptr, *dT = nullptr, *dbg = nullptr, *dpart = nullptr;
  double** dptrs = nullptr;             // [2][2 N_f]: source and destination arrays
  pycool_status st = PYCOOL_OK;
  do {
    if (injected_alloc_failure() ||
        cudaMalloc((void**)&spec, (size_t)2 * nf * half * sizeof(cufftDoubleComplex)) !=
            cudaSuccess ||
        cudaMalloc((void**)&dk, (size_t)nk * sizeof(double)) != cudaSuccess ||
        cudaMalloc((void**)&dT, (size_t)nk * N2 * sizeof(double)) != cudaSuccess ||
        cudaMalloc((void**)&dbg, 16 * sizeof(double) + kLinScratch) != cudaSuccess ||
        cudaMalloc((void**)&dpart, (size_t)2 * nf * kMeanBlocks * sizeof(double)) != cudaSuccess ||
        cudaMalloc((void**)&dptrs, 8 * sizeof(double*)) != cudaSuccess) {
      cudaGetLastError();
      st = PYCOOL_E_NOMEM;
      break;
    }
    if (!own_fft && (cufftSetStream(plans->fwd, s) != CUFFT_SUCCESS ||
                     cufftSetStream(plans->inv, s) != CUFFT_SUCCESS)) {
      st = PYCOOL_E_CUDA;
      break;
    }
    a.k2 = dk;
    a.T = dT;
    a.bg = dbg;
    a.bg_in = dbg + 8;
    cufftDoubleComplex* sphi = spec;
    cufftDoubleComplex* spi = spec + (size_t)nf * half;
    LinSymbol sy;
    std::memset(&sy, 0, sizeof(sy));
    for (int m = 0; m <= hn; ++m) {
      sy.cs[m] = std::cos(2.0 * M_PI * m / n);
      sy.ax4[m] = -(2.0 * (16.0 / 12.0) * sy.cs[m] +
                    2.0 * (-1.0 / 12.0) * std::cos(4.0 * M_PI * m / n));
    }
    linear_k2<<<dim3(hn / 256 + 1, hn + 1, hn + 1), 256, 0, s>>>(sy, hn, cfg->stencil, dk);
    // 1. background: the lattice means (fixed-order sums); the perturbations
    //    (fields minus means) go to the output arrays, which serve as the
    //    transforms' real input (the background never enters a transform)
    double* hptrs[8];
    for (int f = 0; f < nf; ++f) {
      hptrs[f] = const_cast<double*>(phi) + (size_t)f * S;
      hptrs[nf + f] = const_cast<double*>(pi) + (size_t)f * S;
      hptrs[4 + f] = phi_out + (size_t)f * S;
      hptrs[4 + nf + f] = pi_out + (size_t)f * S;
    }
    if (cudaMemcpyAsync(dptrs, hptrs, sizeof(hptrs), cudaMemcpyHostToDevice, s) != cudaSuccess) {
      st = PYCOOL_E_CUDA;
      break;
    }
    linear_means_partial<<<dim3(kMeanBlocks, 2 * nf), 256, 0, s>>>(dptrs, S, dpart);
    linear_means_fold<<<1, 32, 0, s>>>(dpart, 2 * nf, 1.0 / (double)S, dbg + 8);
    linear_subtract<<<152 * 8, 256, 0, s>>>(dptrs, dptrs + 4, S, 2 * nf, dbg + 8);
    // 2. forward transforms of the perturbations (every field), k = 0 cleared
    bool ok = cudaGetLastError() == cudaSuccess;
    if (own_fft)
      ok = ok && fft_forward(phi_out, sphi, n, nf, s) == cudaSuccess &&
           fft_forward(pi_out, spi, n, nf, s) == cudaSuccess;
    else
      ok = ok && cufftExecD2Z(plans->fwd, phi_out, sphi) == CUFFT_SUCCESS &&
           cufftExecD2Z(plans->fwd, pi_out, spi) == CUFFT_SUCCESS;
    if (!ok) {
      st = PYCOOL_E_CUDA;
      break;
    }
    linear_clear_mean<<<1, 32, 0, s>>>(spec, half, nf);
    // 3. growth functions of the classes of k_eff^2
    // 4. every mode: T y(0) / S, k = 0 -> the evolved background
    if (cudaGetLastError() != cudaSuccess || launch_linear_growth(cfg->model, a, dbg + 16, s) != cudaSuccess ||
        launch_linear_apply(nf, spec, half, n, dT, dbg, 1.0 / (double)S, s) != cudaSuccess) {
      st = PYCOOL_E_CUDA;
      break;
    }
    // 5. inverse transforms into the caller's arrays
    if (own_fft)
      ok = fft_inverse(sphi, phi_out, n, nf, s) == cudaSuccess &&
           fft_inverse(spi, pi_out, n, nf, s) == cudaSuccess;
    else
      ok = cufftExecZ2D(plans->inv, sphi, phi_out) == CUFFT_SUCCESS &&
           cufftExecZ2D(plans->inv, spi, pi_out) == CUFFT_SUCCESS;
    if (!ok) {
      st = PYCOOL_E_CUDA;
      break;
    }
    if (cudaMemcpyAsync(background, dbg, (size_t)(2 + 2 * nf) * sizeof(double),
                        cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
      st = PYCOOL_E_CUDA;
  } while (0);
  cudaFree(spec);
  cudaFree(dk);
  cudaFree(dT);
  cudaFree(dbg);
  cudaFree(dpart);
  cudaFree(dptrs);
  return st;
}
