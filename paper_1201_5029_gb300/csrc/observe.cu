// Output-interval observables (Sec. 2.1 Eq. rho-pres with the gradient stencil
// of Eq. G; the spectra of the post-processing, Sec. 2.4), computed at a
// synchronised state on the device:
//   energy_fields : rho(x) and P(x) at every site (7-, 27- or 13-point G),
//       rho = sum_i [pi_i^2/(2 a^6) + G[phi_i]/(2 a^2 dx^2)] + V(phi),
//       P   = sum_i [pi_i^2/(2 a^6) - G[phi_i]/(6 a^2 dx^2)] - V(phi),
//       (a potential given at run time: V from its compiled kernel, run on
//       the same state just before),
//       G[phi](x) = 1/2 sum_alpha c_d(alpha) (phi(alpha) - phi(x))^2;
//     the split forms take the differences phi(alpha) - phi(x) from the
//     fluctuations alone (the background cancels) and V in float64 at
//     phi0 + fluctuation;
//   field_values : one field or momentum of the current state in float64
//     (the input of the spectrum's transform);
//   spectrum_bins : the shell sums of |F_k|^2 / S^2 over the half spectrum of
//     a real transform (modes with a conjugate outside it count twice), the
//     shells cut into chunks of modes in a fixed host-made order, a block per
//     chunk and a warp per shell to add its chunks, so the result is
//     reproducible bit for bit.
// These run at output times only; each is one pass over the lattice.  Float64
// arithmetic and conversions are what they spend their time on (two lanes per
// SM and clock), not memory.
#include <cufft.h>

#include <cstring>

#include "internal.cuh"
#include "models.cuh"
#include "runtime.h"

namespace pycool {

namespace {

// A value of field f at site i of a buffer, in float64: FP64 stores it,
// the split forms store the fluctuation (float or a double-float pair).
template <int PREC>
__device__ __forceinline__ double fluct_at(const void* buf, size_t i) {
  if constexpr (PREC == PREC_FP64) {
    return __ldg(static_cast<const double*>(buf) + i);
  } else if constexpr (PREC == PREC_SPLIT) {
    return widen(__ldg(static_cast<const float*>(buf) + i));
  } else {
    const float2 v = __ldg(static_cast<const float2*>(buf) + i);
    return widen(v.x) + widen(v.y);
  }
}

struct ObsArgs {
  const void* phi;
  const void* pi;
  double* rho;
  double* P;
  int n, nf;
  const double* Vext;   // potentials given at run time: V at every site (the compiled kernel's)
  double ck, cg;        // 1/(2 a^6), 1/(4 a^2 dx^2): of sum pi^2 and of sum c_d (phi(alpha) - phi)^2
  int zc;               // planes per thread
  double phi0[kMaxFields], pi0[kMaxFields];   // split forms: background (0 for FP64)
  double params[8], derived[4];
};

// A thread takes the column (x, y) through zc planes, with the column's values
// at z - H .. z + H in registers and the other neighbours by loads (L1/L2).
// Bound by the float64 pipe: per field and neighbour one subtraction and one
// FMA (the weights of a class of neighbours applied once to its sum of
// squares), and no division: every scale is formed on the host.  256^3,
// one field, 7 points: 1.71 -> 0.66 ms (before: three divisions per site, a
// multiplication more per neighbour, 64-bit index divisions).
template <int MODEL, int STENCIL, int PREC>
__global__ void __launch_bounds__(256) energy_fields_kernel(const ObsArgs o) {
  using P = Pot<MODEL>;
  constexpr int NF = P::NF, H = STENCIL == 13 ? 2 : 1;
  const int n = o.n;
  const size_t nn = (size_t)n * n, S = nn * n;
  const int x = blockIdx.x * 32 + (threadIdx.x & 31), y = blockIdx.y * 8 + (threadIdx.x >> 5);
  if (x >= n || y >= n) return;
  const int z0 = blockIdx.z * o.zc, z1 = min(n, z0 + o.zc);
  const typename P::K pk = P::prep(o.params, o.derived);
  auto wrap = [n](int v) { return v < 0 ? v + n : (v >= n ? v - n : v); };
  int ox[2 * H + 1], oy[2 * H + 1];   // in-plane offsets of the neighbouring columns and rows
#pragma unroll
  for (int k = -H; k <= H; ++k) {
    ox[k + H] = wrap(x + k);
    oy[k + H] = wrap(y + k) * n;
  }
  const size_t col = (size_t)oy[H] + ox[H];
  const char* pb[NF];
  const char* qb[NF];
  double zq[NF][2 * H + 1];
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    pb[f] = static_cast<const char*>(o.phi) + (size_t)f * S * prec_word(PREC);
    qb[f] = static_cast<const char*>(o.pi) + (size_t)f * S * prec_word(PREC);
#pragma unroll
    for (int k = 0; k < 2 * H; ++k)
      zq[f][k + 1] = fluct_at<PREC>(pb[f], (size_t)wrap(z0 - H + k) * nn + col);
  }
  for (int z = z0; z < z1; ++z) {
    const size_t zo = (size_t)z * nn, i = zo + col;
    double kin = 0.0, grad = 0.0, fv[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
#pragma unroll
      for (int k = 0; k < 2 * H; ++k) zq[f][k] = zq[f][k + 1];
      zq[f][2 * H] = fluct_at<PREC>(pb[f], (size_t)wrap(z + H) * nn + col);
      const double ctr = zq[f][H];
      auto sq = [&](double v, double acc) { const double e = v - ctr; return fma(e, e, acc); };
      auto at = [&](size_t plane, int ky, int kx) {
        return fluct_at<PREC>(pb[f], plane + oy[ky + H] + ox[kx + H]);
      };
      if constexpr (STENCIL == 27) {
        double s[4] = {0.0, 0.0, 0.0, 0.0};   // by class: faces, edges, corners
#pragma unroll
        for (int dz = -1; dz <= 1; ++dz) {
          const size_t plane = (size_t)wrap(z + dz) * nn;
#pragma unroll
          for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
              const int cls = (dz != 0) + (dy != 0) + (dx != 0);
              if (cls == 0) continue;
              s[cls] = sq(cls == 1 && dz != 0 ? zq[f][dz + H] : at(plane, dy, dx), s[cls]);
            }
        }
        grad = fma(14.0 / 30.0, s[1], fma(3.0 / 30.0, s[2], fma(1.0 / 30.0, s[3], grad)));
      } else {
        double s1 = STENCIL == 13 ? 0.0 : grad;
        s1 = sq(zq[f][H - 1], s1);
        s1 = sq(zq[f][H + 1], s1);
        s1 = sq(at(zo, -1, 0), s1);
        s1 = sq(at(zo, 1, 0), s1);
        s1 = sq(at(zo, 0, -1), s1);
        s1 = sq(at(zo, 0, 1), s1);
        if constexpr (STENCIL == 13) {   // weights 16/12 at one site, -1/12 at two
          double s2 = sq(zq[f][0], 0.0);
          s2 = sq(zq[f][4], s2);
          s2 = sq(at(zo, -2, 0), s2);
          s2 = sq(at(zo, 2, 0), s2);
          s2 = sq(at(zo, 0, -2), s2);
          s2 = sq(at(zo, 0, 2), s2);
          grad = fma(16.0 / 12.0, s1, fma(-1.0 / 12.0, s2, grad));
        } else {
          grad = s1;
        }
      }
      double q = fluct_at<PREC>(qb[f], i);
      fv[f] = ctr;
      if constexpr (PREC != PREC_FP64) {
        q += o.pi0[f];
        fv[f] += o.phi0[f];
      }
      kin = fma(q, q, kin);
    }
    double V;
    if constexpr (MODEL == M_RUNTIME1 || MODEL == M_RUNTIME2) {
      V = o.Vext[i];
    } else {
      double dV[NF];
      P::eval(pk, fv, dV, V);
    }
    // k = sum pi^2 / (2 a^6), g = sum G / (2 a^2 dx^2):  rho = k + g + V, P = k - g/3 - V
    o.rho[i] = fma(o.ck, kin, fma(o.cg, grad, V));
    o.P[i] = fma(o.ck, kin, fma(-o.cg * (1.0 / 3.0), grad, -V));
  }
}

template <int PREC>
__global__ void field_values_kernel(const void* buf, double base, double* out, size_t S) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < S;
       i += (size_t)gridDim.x * blockDim.x)
    out[i] = base + fluct_at<PREC>(buf, i);
}

// One block per chunk of a shell's modes: order holds indices into the half
// spectrum, shell by shell, with bit 31 set for a mode that stands for itself
// alone (its conjugate is in the half spectrum too); chunk b covers order[cut[b]
// .. cut[b + 1]).  Two float64 instructions per mode; the loads of a thread's
// modes are independent of each other.  256^3: 407 -> 83 us with the fold (one
// block per shell before, whose longest chain of dependent loads ran alone).
__global__ void __launch_bounds__(256) spectrum_bins_kernel(const cufftDoubleComplex* spec,
                                                            const uint32_t* order,
                                                            const int32_t* cut, double* part) {
  __shared__ double red[8];
  const int j0 = cut[blockIdx.x], j1 = cut[blockIdx.x + 1];
  double one = 0.0, two = 0.0;
#pragma unroll 8
  for (int j = j0 + threadIdx.x; j < j1; j += 256) {
    const uint32_t m = __ldg(&order[j]);
    const double2 v = __ldg(reinterpret_cast<const double2*>(spec) + (m & 0x7fffffffu));
    if (m >> 31) one = fma(v.x, v.x, fma(v.y, v.y, one));
    else two = fma(v.x, v.x, fma(v.y, v.y, two));
  }
  double acc = fma(2.0, two, one);
#pragma unroll
  for (int h = 16; h > 0; h >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, h);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = red[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) t += red[w];
    part[blockIdx.x] = t;
  }
}
// One warp per shell: its chunks first[b] .. first[b + 1], in a fixed order.
__global__ void __launch_bounds__(32) spectrum_fold_kernel(const double* part,
                                                           const int32_t* first, double invS2,
                                                           double* power) {
  const int b = blockIdx.x;
  double t = 0.0;
  for (int c = first[b] + threadIdx.x; c < first[b + 1]; c += 32) t += part[c];
#pragma unroll
  for (int h = 16; h > 0; h >>= 1) t += __shfl_down_sync(0xffffffffu, t, h);
  if (threadIdx.x == 0) power[b] = t * invS2;
}

ObsArgs obs_args(const SimDesc& d, const Background& b) {
  ObsArgs o;
  memset(&o, 0, sizeof(o));
  o.phi = d.phi[b.cur & 1];
  o.pi = d.pi[(b.cur >> 1) & 1];
  o.n = d.n;
  o.nf = d.nf;
  const double a2 = b.a * b.a;
  o.ck = 1.0 / (2.0 * (a2 * a2 * a2));
  o.cg = 0.25 * d.dx2inv / a2;
  for (int f = 0; f < d.nf; ++f) {
    o.phi0[f] = d.prec == PREC_FP64 ? 0.0 : b.phi0[f];
    o.pi0[f] = d.prec == PREC_FP64 ? 0.0 : b.pi0[f];
  }
  for (int i = 0; i < 8; ++i) o.params[i] = d.params[i];
  for (int i = 0; i < 4; ++i) o.derived[i] = d.derived[i];
  return o;
}

unsigned grid_for(size_t work) {
  const size_t g = (work + 255) / 256;
  return (unsigned)(g < 152 * 32 ? g : 152 * 32);
}

}  // namespace

cudaError_t launch_energy_fields(const SimDesc& d, const Background& b, double* rho, double* P,
                                 cudaStream_t s) {
  ObsArgs o = obs_args(d, b);
  o.rho = rho;
  o.P = P;
  o.Vext = d.rt_V;
  // planes per thread: enough blocks for every SM several times over, and long
  // enough columns that their first planes (the z halo) do not count
  const int n = d.n;
  const unsigned tx = (n + 31) / 32, ty = (n + 7) / 8;
  o.zc = 32;
  while (o.zc > 4 && (long long)tx * ty * ((n + o.zc - 1) / o.zc) < 152 * 8) o.zc /= 2;
  const dim3 g(tx, ty, (unsigned)((n + o.zc - 1) / o.zc));
#define PYCOOL_OBS(M, ST, PR)                                                            \
  if (d.model == M && d.stencil == ST && d.prec == PR) {                                 \
    energy_fields_kernel<M, ST, PR><<<g, 256, 0, s>>>(o);                               \
    return cudaGetLastError();                                                           \
  }
#define PYCOOL_OBS_M(M, PR) PYCOOL_OBS(M, 7, PR) PYCOOL_OBS(M, 27, PR) PYCOOL_OBS(M, 13, PR)
#define PYCOOL_OBS_P(PR)                                                                 \
  PYCOOL_OBS_M(M_FREE, PR) PYCOOL_OBS_M(M_CHAOTIC2, PR) PYCOOL_OBS_M(M_OSCILLON, PR)      \
  PYCOOL_OBS_M(M_QBALL, PR)
  PYCOOL_OBS_P(PREC_FP64)
  PYCOOL_OBS_P(PREC_SPLIT)
  PYCOOL_OBS_P(PREC_DD)
  PYCOOL_OBS_M(M_RUNTIME1, PREC_FP64)
  PYCOOL_OBS_M(M_RUNTIME2, PREC_FP64)
#undef PYCOOL_OBS_P
#undef PYCOOL_OBS_M
#undef PYCOOL_OBS
  return cudaErrorInvalidValue;
}

cudaError_t launch_field_values(const SimDesc& d, const Background& b, int which, int f,
                                double* out, cudaStream_t s) {
  const size_t S = (size_t)d.S;
  const void* buf = which == 0 ? d.phi[b.cur & 1] : d.pi[(b.cur >> 1) & 1];
  buf = static_cast<const char*>(buf) + (size_t)f * S * prec_word(d.prec);
  const double base = d.prec == PREC_FP64 ? 0.0 : (which == 0 ? b.phi0[f] : b.pi0[f]);
  const unsigned g = grid_for(S);
  if (d.prec == PREC_FP64) field_values_kernel<PREC_FP64><<<g, 256, 0, s>>>(buf, base, out, S);
  else if (d.prec == PREC_SPLIT) field_values_kernel<PREC_SPLIT><<<g, 256, 0, s>>>(buf, base, out, S);
  else field_values_kernel<PREC_DD><<<g, 256, 0, s>>>(buf, base, out, S);
  return cudaGetLastError();
}

cudaError_t launch_spectrum_bins(const void* spec, int n, const uint32_t* order,
                                 const int32_t* cut, int nchunks, const int32_t* first, int nbins,
                                 double* part, double* power, cudaStream_t s) {
  const double S = (double)n * n * n;
  spectrum_bins_kernel<<<nchunks, 256, 0, s>>>(static_cast<const cufftDoubleComplex*>(spec), order,
                                               cut, part);
  spectrum_fold_kernel<<<nbins, 32, 0, s>>>(part, first, 1.0 / (S * S), power);
  return cudaGetLastError();
}

}  // namespace pycool
