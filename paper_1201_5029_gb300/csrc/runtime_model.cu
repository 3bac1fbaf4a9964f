// Potentials given at run time.  PyCOOL turns the potential strings of a
// model file into CUDA kernels with SymPy and jinja2 templates, compiled by
// PyCUDA, and writes them out for inspection (Sec. 2.4).  Here the caller
// gives the potential and its derivatives as C expressions in the fields f0,
// f1 and the parameters p[0..7] (pycool_model_define); NVRTC compiles them
// into one elementwise kernel for the device the library runs on, which a
// stage launches between the library's own drift and kick kernels
// (sweep.cuh: rt_drift, rt_kick).  The generated source can be read back
// (pycool_model_source).
#include <cuda_runtime.h>
#include <nvrtc.h>

#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "../../include/pycool.h"
#include "persist_plain.cuh"
#include "runtime.h"

#define PYCOOL_API extern "C" __attribute__((visibility("default")))

namespace pycool {

namespace {

struct RtModel {
  int nf = 0;
  std::string source;
  cudaLibrary_t lib = nullptr;
  cudaKernel_t kern = nullptr;
};

std::mutex g_rt_mu;
std::vector<RtModel> g_rt;   // entry i is model id kRuntimeModelBase + i

struct RtParams {
  double p[8];
};

std::string make_source(int nf, const char* V, const char* const* dV) {
  std::string s =
      "// generated by pycool_model_define: V and dV/dphi_i of a potential given at run time\n"
      "struct RtParams { double p[8]; };\n"
      "extern \"C\" __global__ void pycool_model_kernel(const double* __restrict__ phis,\n"
      "    double* __restrict__ dV, double* __restrict__ V, long long S, const RtParams prm) {\n"
      "  const double* p = prm.p;\n"
      "  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < S;\n"
      "       i += (long long)gridDim.x * blockDim.x) {\n"
      "    const double f0 = phis[i];\n";
  if (nf == 2) s += "    const double f1 = phis[S + i];\n";
  s += "    V[i] = (" + std::string(V) + ");\n";
  s += "    dV[i] = (" + std::string(dV[0]) + ");\n";
  if (nf == 2) s += "    dV[S + i] = (" + std::string(dV[1]) + ");\n";
  s += "  }\n}\n";
  return s;
}

// The kick of a stage: one stage of the plain staging over each block's units
// (one block per SM), with V' and V read from the compiled kernel's arrays, then
// the per-stage kernels' block finish.  Bound by the float64 pipe: ten
// instructions per two-field site (128^3: 51 % of it; 16 warps and a barrier of
// all of them per plane do not cover the rest).
template <int MODEL, int STENCIL>
__global__ void __launch_bounds__(kPThreads, 1) rt_kick(const LaunchTable tab) {
  using C = Ctx<MODEL, PREC_FP64>;
  using SL = typename C::SL;
  constexpr int NF = C::NF, NQ = SL::NQ, H = halo_of<STENCIL>();
  using RG = PlainRing<NF, NQ, H>;
  extern __shared__ __align__(128) unsigned char dsm[];
  __shared__ __align__(8) uint64_t dbar[RG::NDRIFT];
  __shared__ __align__(64) SimDesc s_desc;
  __shared__ int4 s_units[kMaxPUnits];
  __shared__ double sout[NQ];
  __shared__ uint32_t s_wmax[kPWarps][2 * NF], s_bmax[2 * NF];
  __shared__ C s_ctx;
  __shared__ int s_last, s_bad;
  const SimDesc* dg = tab.desc[0];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int mode = dg->bg->mode;
  if (mode == MODE_IDLE) return;
  const int ubeg = dg->rt_uoff[blockIdx.x];
  PShared sm;
  sm.d = &s_desc;
  sm.ring = dsm;
  sm.kahan = nullptr;
  sm.drift = nullptr;
  sm.red = reinterpret_cast<double*>(dsm + RG::RING_BYTES);
  sm.full = sm.empty = nullptr;
  sm.dbar = dbar;
  sm.units = s_units;
  sm.nunits = min(dg->rt_uoff[blockIdx.x + 1] - ubeg, kMaxPUnits);   // host: <= kMaxPUnits
  sm.issued = nullptr;
  sm.limit = kWaitLimit;
  for (int i = tid; i < (int)(sizeof(SimDesc) / 8); i += kPThreads)
    reinterpret_cast<unsigned long long*>(&s_desc)[i] =
        reinterpret_cast<const unsigned long long*>(dg)[i];
  if (tid < sm.nunits) s_units[tid] = dg->rt_units[ubeg + tid];
  if (tid == 0) {
    for (int b = 0; b < RG::NDRIFT; ++b) mbar_init(&dbar[b], kPWarps);
    fence_mbar_init();
    s_bad = 0;
  }
  __syncthreads();
  const SimDesc& d = s_desc;
  const Background& bgr = *d.bg;
  const int n = d.n, ib = bgr.cur;
  plain_prefetch<MODEL, NQ, H>(n, sm, ib, 0u);   // while one thread ...
  if (tid == 0) {
    s_ctx.init(bgr, d, mode);
    s_ctx.set_fix(bgr.amax, fix_headroom<STENCIL>());
  }
  __syncthreads();
  double ps[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) ps[q] = 0.0;
  HiMax<NF> hm;
  hm.zero();
  bool ok = true;
  by_mode(mode, s_ctx.fx[0] != 0, [&](auto fix_c, auto mode_c) {
    ok = stage_plain<MODEL, STENCIL, decltype(mode_c)::value, decltype(fix_c)::value>(
        n, s_ctx, sm, 0u, ib, ps, hm);
  });
  cp_async_wait<0>();
  if (!ok) s_bad = 1;
#pragma unroll
  for (int i = 0; i < 2 * NF; ++i) {
    const uint32_t m = __reduce_max_sync(0xffffffffu, hm.v[i]);
    if (lane == 0) s_wmax[warp][i] = m;
  }
  __syncthreads();
  if (s_bad) {   // a wait gave up: recorded, and the stage is not finished
    if (tid == 0) atomicOr(d.fault, 1);
    return;
  }
  constexpr uint32_t kSweepLive = (1u << SL::PI2) | (1u << SL::PHID) | (1u << SL::V);
  block_sum<NQ, kPWarps>(ps, sm.red, sout, mode == MODE_SWEEP ? kSweepLive : 0xffffffffu);
  if (tid < 2 * NF) {
    uint32_t m = 0u;
#pragma unroll
    for (int w = 0; w < kPWarps; ++w) m = max(m, s_wmax[w][tid]);
    s_bmax[tid] = m;
  }
  __syncthreads();
  finish_block<MODEL, PREC_FP64>(s_ctx, d, mode, blockIdx.x, sout, &s_last, s_bmax);
}

template <int MODEL, int STENCIL>
cudaError_t launch_rt_kick(const LaunchTable& t, int grid, cudaStream_t s) {
  constexpr int NF = Pot<MODEL>::NF;
  constexpr int smem =
      PlainRing<NF, Slots<NF, PREC_FP64>::NQ, halo_of<STENCIL>()>::SMEM_BYTES;
  if (grid == 0)   // ahead of any stream capture
    return cudaFuncSetAttribute(rt_kick<MODEL, STENCIL>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  rt_kick<MODEL, STENCIL><<<grid, kPThreads, smem, s>>>(t);
  return cudaGetLastError();
}

}  // namespace

int runtime_model_nfields(int id) {
  std::lock_guard<std::mutex> lk(g_rt_mu);
  const int i = id - kRuntimeModelBase;
  return (i >= 0 && i < (int)g_rt.size()) ? g_rt[i].nf : -1;
}

// The compiled potential of a runtime-model simulation at the fields `phis`
// (N_f n^3 float64 values): V' into d.rt_dV, V into d.rt_V.
cudaError_t launch_runtime_potential(const SimDesc& d, const double* phis, cudaStream_t s) {
  cudaKernel_t kern = nullptr;
  {
    std::lock_guard<std::mutex> lk(g_rt_mu);
    if (d.rt_index < 0 || d.rt_index >= (int)g_rt.size()) return cudaErrorInvalidValue;
    kern = g_rt[d.rt_index].kern;
  }
  double* dV = d.rt_dV;
  double* V = d.rt_V;
  long long S = (long long)d.S;
  RtParams prm;
  for (int i = 0; i < 8; ++i) prm.p[i] = d.params[i];
  void* args[] = {(void*)&phis, (void*)&dV, (void*)&V, (void*)&S, (void*)&prm};
  return cudaLaunchKernel((const void*)kern, dim3(152 * 8), dim3(256), args, 0, s);
}

// One stage of a runtime-model simulation: drift, the compiled potential, kick.
cudaError_t launch_runtime_stage(const SimDesc& d, const LaunchTable& t, int grid,
                                 cudaStream_t s) {
  {
    std::lock_guard<std::mutex> lk(g_rt_mu);
    if (d.rt_index < 0 || d.rt_index >= (int)g_rt.size()) return cudaErrorInvalidValue;
  }
  if (grid != 0) {   // 0: set the kernel's attributes only
    const unsigned eg = 152;
    if (d.model == M_RUNTIME1) rt_drift<M_RUNTIME1><<<eg, kRtDriftThreads, 0, s>>>(t);
    else rt_drift<M_RUNTIME2><<<eg, kRtDriftThreads, 0, s>>>(t);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_runtime_potential(d, d.rt_phis, s);
    if (e != cudaSuccess) return e;
  }
#define PYCOOL_RT(M, ST)                                              \
  if (d.model == M && d.stencil == ST) {                              \
    return launch_rt_kick<M, ST>(t, grid, s);                         \
  }
  PYCOOL_RT(M_RUNTIME1, 7) PYCOOL_RT(M_RUNTIME1, 27) PYCOOL_RT(M_RUNTIME1, 13)
  PYCOOL_RT(M_RUNTIME2, 7) PYCOOL_RT(M_RUNTIME2, 27) PYCOOL_RT(M_RUNTIME2, 13)
#undef PYCOOL_RT
  return cudaErrorInvalidValue;
}

}  // namespace pycool

using namespace pycool;

PYCOOL_API pycool_status pycool_model_define(int32_t nf, const char* V, const char* const* dV,
                                             int32_t* model_id) {
  if (!model_id || (nf != 1 && nf != 2) || !V || !dV || !dV[0] || (nf == 2 && !dV[1]))
    return PYCOOL_E_INVALID;
  {
    std::lock_guard<std::mutex> lk(g_rt_mu);
    if ((int)g_rt.size() >= kRuntimeModelMax) return PYCOOL_E_NOMEM;
  }
  RtModel m;
  m.nf = nf;
  m.source = make_source(nf, V, dV);
  nvrtcProgram prog;
  if (nvrtcCreateProgram(&prog, m.source.c_str(), "pycool_model.cu", 0, nullptr, nullptr) !=
      NVRTC_SUCCESS)
    return PYCOOL_E_CUDA;
  const char* opts[] = {"--gpu-architecture=sm_103a", "--std=c++17"};
  const nvrtcResult cr = nvrtcCompileProgram(prog, 2, opts);
  if (cr != NVRTC_SUCCESS) {
    size_t n = 0;
    nvrtcGetProgramLogSize(prog, &n);
    std::string log(n, '\0');
    if (n) nvrtcGetProgramLog(prog, &log[0]);
    std::fprintf(stderr, "pycool_model_define: the expressions do not compile:\n%s\n",
                 log.c_str());
    nvrtcDestroyProgram(&prog);
    return PYCOOL_E_INVALID;
  }
  size_t cubin_size = 0;
  std::vector<char> cubin;
  if (nvrtcGetCUBINSize(prog, &cubin_size) != NVRTC_SUCCESS || cubin_size == 0) {
    nvrtcDestroyProgram(&prog);
    return PYCOOL_E_CUDA;
  }
  cubin.resize(cubin_size);
  const nvrtcResult gr = nvrtcGetCUBIN(prog, cubin.data());
  nvrtcDestroyProgram(&prog);
  if (gr != NVRTC_SUCCESS) return PYCOOL_E_CUDA;
  if (cudaLibraryLoadData(&m.lib, cubin.data(), nullptr, nullptr, 0, nullptr, nullptr, 0) !=
          cudaSuccess ||
      cudaLibraryGetKernel(&m.kern, m.lib, "pycool_model_kernel") != cudaSuccess) {
    cudaGetLastError();
    if (m.lib) cudaLibraryUnload(m.lib);
    return PYCOOL_E_CUDA;
  }
  std::lock_guard<std::mutex> lk(g_rt_mu);
  g_rt.push_back(m);
  *model_id = kRuntimeModelBase + (int32_t)g_rt.size() - 1;
  return PYCOOL_OK;
}

PYCOOL_API pycool_status pycool_model_source(int32_t model_id, char* buf, size_t cap,
                                             size_t* len) {
  std::lock_guard<std::mutex> lk(g_rt_mu);
  const int i = model_id - kRuntimeModelBase;
  if (i < 0 || i >= (int)g_rt.size()) return PYCOOL_E_INVALID;
  const std::string& src = g_rt[i].source;
  if (len) *len = src.size();
  if (buf) {
    if (cap < src.size() + 1) return PYCOOL_E_INVALID;
    std::memcpy(buf, src.c_str(), src.size() + 1);
  }
  return PYCOOL_OK;
}
