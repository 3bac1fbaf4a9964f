// The persistent evolve kernel itself (see persist.cuh for what a stage does):
// start, the stages' block sums, the grid barrier and the scalar chain between
// stages, and the launch helper.
#pragma once

#include "persist_plain.cuh"

namespace pycool {

// The shared-memory ring of an instance: VX > 0 the TMA staging with VX sites
// per lane, VX = 0 the plain staging (persist_plain.cuh, FP64).
template <int PREC, int NF, int VX, int NQ, int H>
struct RingOf { using type = PRing<PREC, NF, VX, NQ, H>; };
template <int NF, int NQ, int H>
struct RingOf<PREC_FP64, NF, 0, NQ, H> { using type = PlainRing<NF, NQ, H>; };

// ---------------------------------------------------------------------------
// The kernel.
// ---------------------------------------------------------------------------
template <int MODEL, int STENCIL, int PREC, int VX>
__global__ void __launch_bounds__(kPThreads, 1) evolve_persist(const __grid_constant__ PParams p) {
  using C = Ctx<MODEL, PREC>;
  using SL = typename C::SL;
  constexpr int NQ = SL::NQ;
  constexpr int NF = C::NF;
  constexpr bool CORNERS = StencilW<STENCIL>::kCorners;
  constexpr int H = halo_of<STENCIL>();
  constexpr bool PLAIN = VX == 0;
  static_assert(STENCIL != 13 || PREC != PREC_SPLIT, "the 13-point stencil: FP64 and split-DD");
  using RG = typename RingOf<PREC, NF, VX, NQ, H>::type;
  constexpr int NSLOT = RG::NSLOT, LEAD = RG::LEAD, PRE = RG::PRE;
  static_assert(RG::FOLD <= kPWarps, "one warp per reduced quantity");
  static_assert(PREC == PREC_SPLIT || (size_t)kMaxPBlocks * kNQ * 8 <= (size_t)NQ * kPThreads * 8,
                "the rows of every block fit the reduction scratch");

  extern __shared__ __align__(128) unsigned char dsm[];
  __shared__ __align__(8) uint64_t full[NSLOT], empty[NSLOT], foldbar, dbar[RG::NDRIFT];
  // background and stage coefficients, double-buffered: at a stage boundary
  // one thread derives the next coefficients while another does the rest of
  // the background bookkeeping
  __shared__ __align__(16) Background sbv[2];
  __shared__ C sctxv[2];
  // formed during the fold: the sums-to-kick coefficients of this stage and
  // the sums-independent half of the next stage's scalar half-steps
  __shared__ SumCoef<NF> s_sc;
  __shared__ PreCoef s_qn;
  __shared__ double s_p0[2 * NF];   // split form: the next stage's re-centred background
  // the scalar chain between stages reads the descriptor many times; the
  // ring leaves little L1, so it is kept in shared memory
  __shared__ __align__(64) SimDesc s_desc;
  __shared__ double sums[kNQ];
  __shared__ uint32_t s_wmax[kPWarps][2 * NF];   // FP64: each warp's largest |phi|, |pi| ...
  __shared__ uint32_t s_amax[2 * kMaxFields];    // ... and the lattice's (Background::amax)
  __shared__ int4 s_units[kMaxPUnits];
  __shared__ uint32_t s_issued[NSLOT];
  __shared__ int s_bad;
  __shared__ int s_fold;   // parity of a rows copy issued and not yet folded; -1: none

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const SimDesc& d = s_desc;
  const int G = p.g.G;
  static_assert(sizeof(SimDesc) % 8 == 0, "descriptor copied as 8-byte words");
  for (int i = tid; i < (int)(sizeof(SimDesc) / 8); i += kPThreads)
    reinterpret_cast<unsigned long long*>(&s_desc)[i] =
        __ldg(reinterpret_cast<const unsigned long long*>(p.d) + i);
  PShared sm;
  sm.d = &s_desc;
  sm.ring = dsm;
  sm.kahan = reinterpret_cast<float2*>(dsm + RG::RING_BYTES);
  sm.drift = reinterpret_cast<double*>(dsm + RG::RING_BYTES);
  sm.red = reinterpret_cast<double*>(dsm + RG::RING_BYTES) + RG::DRIFT_WORDS;
  sm.full = full;
  sm.empty = empty;
  sm.dbar = dbar;
  sm.units = s_units;
  sm.issued = s_issued;
  sm.limit = p.wait_limit;
  const int ubeg = __ldg(&p.uoff[blockIdx.x]);
  sm.nunits = min(__ldg(&p.uoff[blockIdx.x + 1]) - ubeg, kMaxPUnits);   // host: <= kMaxPUnits

  if (tid == 0) {
    for (int s = 0; s < NSLOT; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], kPWarps);
    }
    mbar_init(&foldbar, 1);
    for (int b = 0; b < RG::NDRIFT; ++b) mbar_init(&dbar[b], kPWarps);
    fence_mbar_init();
    s_bad = 0;
    s_fold = -1;
  }
  if (tid < NSLOT) s_issued[tid] = 0;
  if (!PLAIN && tid < 6) {   // bring the tensor maps into the descriptor cache
    const CUtensorMap* m = &p.tm[tid];
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
  }
  if (tid < sm.nunits) s_units[tid] = p.units[ubeg + tid];   // this block's units, in order
  static_assert(sizeof(Background) % 8 == 0, "background copied as 8-byte words");
  if (tid < (int)(sizeof(Background) / 8))
    reinterpret_cast<unsigned long long*>(&sbv[0])[tid] =
        __ldcg(reinterpret_cast<const unsigned long long*>(p.bg) + tid);
  __syncthreads();
  if (sbv[0].error) return;   // a stopped simulation stays stopped (same in every block)
  if (tid == 0) {
    sbv[0].sweeps_left = p.nsweeps;
    sbv[0].mode = p.nsweeps > 0 ? MODE_SWEEP : MODE_FLUSH;
  }
  int cb = 0;   // current buffer of sbv / sctxv
  uint32_t np = 0;
  for (int i = 0; i < sm.nunits; ++i) np += (uint32_t)s_units[i].w;
  uint32_t gq = 0;
  const long long K = p.nsweeps;
  // the launch's last pass: the flush (k == K), or, for a launch that leaves
  // the merged stage boundary pending for the next launch (p.flush == 0), the
  // last stage sweep; the Background written back is then a sweep's, as after
  // a per-stage launch
  const long long KL = p.flush ? K : K - 1;
  bool fault = false;
  int ib = sbv[0].cur;
  // stage 0: its first planes are in flight while one thread derives the
  // scalar coefficients (the FP64 chain of the merged half-stages)
  {
    if constexpr (PLAIN) {
      plain_prefetch<MODEL, NQ, H>(p.g.n, sm, ib, gq);
    } else {
      for (int l = kPWarps - 1 - warp; l < LEAD; l += kPWarps)   // warp 15 - l issues plane l
        prefetch_plane<PREC, NF, VX, CORNERS, NSLOT, H>(p, sm, ib, gq, l);
    }
    if (tid == 0) {
      sctxv[0].init(sbv[0], d, K > 0 ? MODE_SWEEP : MODE_FLUSH);
      if constexpr (PREC == PREC_FP64) sctxv[0].set_fix(sbv[0].amax, fix_headroom<STENCIL>());
    }
    __syncthreads();
    fault = s_bad != 0;
  }
  for (long long k = 0; k <= KL && !fault; ++k) {
    const int mode = (k < K) ? MODE_SWEEP : MODE_FLUSH;
    const C cx = sctxv[cb];
    // @stage-start

    // ---- the sweep (per-thread sums) ----
    bool ok = true;
    double accd[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) accd[q] = 0.0;
    HiMax<NF> hm;   // FP64: largest |phi|, |pi| put out
    hm.zero();
    if constexpr (PREC == PREC_FP64) {
      const bool fix = cx.fx[0] != 0;
      auto stage = [&](auto mode_c, auto fix_c) {
        constexpr int MD = decltype(mode_c)::value;
        constexpr bool FX = decltype(fix_c)::value;
        if constexpr (PLAIN)
          return stage_plain<MODEL, STENCIL, MD, FX>(p.g.n, cx, sm, gq, ib, accd, hm);
        else if constexpr (STENCIL == 13)
          return stage_fp64_wide<MODEL, VX, MD, FX>(p, cx, sm, gq, ib, accd, hm);
        else
          return stage_fp64<MODEL, STENCIL, VX, MD, FX>(p, cx, sm, gq, ib, accd, hm);
      };
      using MS = std::integral_constant<int, MODE_SWEEP>;
      using MF = std::integral_constant<int, MODE_FLUSH>;
      if (mode == MODE_SWEEP)
        ok = fix ? stage(MS{}, std::true_type{}) : stage(MS{}, std::false_type{});
      else
        ok = fix ? stage(MF{}, std::true_type{}) : stage(MF{}, std::false_type{});
    } else if constexpr (STENCIL == 13) {
      ok = (mode == MODE_SWEEP) ? stage_wide_dd<MODEL, VX, MODE_SWEEP>(p, cx, sm, gq, ib)
                                : stage_wide_dd<MODEL, VX, MODE_FLUSH>(p, cx, sm, gq, ib);
      const dd* tot = reinterpret_cast<const dd*>(sm.red) + tid;
#pragma unroll
      for (int q = 0; q < NQ; ++q) accd[q] = (double)tot[q * kPThreads];
    } else if constexpr (PREC == PREC_DD) {
      ok = (mode == MODE_SWEEP) ? stage_dd<MODEL, STENCIL, VX, MODE_SWEEP>(p, cx, sm, gq, ib)
                                : stage_dd<MODEL, STENCIL, VX, MODE_FLUSH>(p, cx, sm, gq, ib);
      // this thread's stage sums, from its own scratch slots (overwritten below)
      const dd* tot = reinterpret_cast<const dd*>(sm.red) + tid;
#pragma unroll
      for (int q = 0; q < NQ; ++q) accd[q] = (double)tot[q * kPThreads];
    } else {
      // the Q-ball's difference forms have a branch for a background at the
      // origin; a stage whose background is away from it runs without the test
      // (7-point stencil: the 27-point one would spill with both instances)
      if constexpr (MODEL == M_QBALL && !CORNERS) {
        if (!cx.sk.direct)
          ok = (mode == MODE_SWEEP)
                   ? stage_split<MODEL, STENCIL, VX, MODE_SWEEP, true>(p, cx, sm, gq, ib)
                   : stage_split<MODEL, STENCIL, VX, MODE_FLUSH, true>(p, cx, sm, gq, ib);
        else
          ok = (mode == MODE_SWEEP) ? stage_split<MODEL, STENCIL, VX, MODE_SWEEP>(p, cx, sm, gq, ib)
                                    : stage_split<MODEL, STENCIL, VX, MODE_FLUSH>(p, cx, sm, gq, ib);
      } else {
        ok = (mode == MODE_SWEEP) ? stage_split<MODEL, STENCIL, VX, MODE_SWEEP>(p, cx, sm, gq, ib)
                                  : stage_split<MODEL, STENCIL, VX, MODE_FLUSH>(p, cx, sm, gq, ib);
      }
    }
    if (!ok) atomicOr(&s_bad, 1);
    gq += np;
    // global stores of this stage will be read by TMA (async proxy) next stage
    if constexpr (!PLAIN) fence_proxy_async_global();
    __syncthreads();
    // @units-done
    if (s_bad) { fault = true; break; }

    // ---- block sums: one warp per live quantity over the 512 threads' values, fixed order ----
    const bool sweep = mode == MODE_SWEEP;
    const int nl = sweep ? LiveSlots<NF, PREC>::SWEEP : NQ;   // live quantities
    const int slot = LiveSlots<NF, PREC>::slot(warp, sweep);  // of this warp (warp < nl)
    if (tid < kNQ) sums[tid] = 0.0;
    if constexpr (PREC != PREC_SPLIT) {
      double* red = sm.red;
      if (PREC == PREC_FP64 && sweep) {
        red[tid] = accd[SL::PHID - NF];   // PI2
        red[kPThreads + tid] = accd[SL::PHID];
        red[2 * kPThreads + tid] = accd[SL::V];
      } else {
#pragma unroll
        for (int q = 0; q < NQ; ++q)
          if (q < nl) red[q * kPThreads + tid] = accd[q];
      }
      if constexpr (PREC == PREC_FP64) {
#pragma unroll
        for (int i = 0; i < 2 * NF; ++i) {
          const uint32_t m = __reduce_max_sync(0xffffffffu, hm.v[i]);
          if (lane == 0) s_wmax[warp][i] = m;
        }
      }
      __syncthreads();
      if (warp < nl) {
        // 16 values per lane summed as a pairwise tree (depth 4: FP64 latency is long)
        double x[kPThreads / 32];
#pragma unroll
        for (int r = 0; r < kPThreads / 32; ++r) x[r] = red[warp * kPThreads + lane + 32 * r];
#pragma unroll
        for (int w = kPThreads / 64; w >= 1; w >>= 1)
#pragma unroll
          for (int r = 0; r < w; ++r) x[r] = x[2 * r] + x[2 * r + 1];
        double v = x[0];
#pragma unroll
        for (int h = 16; h >= 1; h >>= 1) v += __shfl_down_sync(0xffffffffu, v, h);
        if (lane == 0) {
          reinterpret_cast<double*>(p.rows)[((size_t)(k & 1) * G + blockIdx.x) * kNQ + slot] = v;
          fence_proxy_async_global();   // the rows are read back by bulk copies
        }
      } else if (PREC == PREC_FP64 && warp == nl) {
        // the block's largest |phi| and |pi| of field f in the row's slot kNQ - 2 + f
        static_assert(PREC != PREC_FP64 || NQ <= kNQ - kMaxFields, "free slots of a row");
        uint32_t m[2 * NF];
#pragma unroll
        for (int i = 0; i < 2 * NF; ++i)
          m[i] = __reduce_max_sync(0xffffffffu, s_wmax[lane % kPWarps][i]);
        if (lane == 0) {
          uint2* row = reinterpret_cast<uint2*>(
              reinterpret_cast<double*>(p.rows) + ((size_t)(k & 1) * G + blockIdx.x) * kNQ +
              kNQ - kMaxFields);
#pragma unroll
          for (int f = 0; f < NF; ++f) row[f] = make_uint2(m[2 * f], m[2 * f + 1]);
          fence_proxy_async_global();
        }
      }
    } else {
      if (warp < nl) {
        float hi = 0.f, lo = 0.f;
#pragma unroll
        for (int r = 0; r < kKahanGroups / 32; ++r) {
          const float2 v = sm.kahan[warp * kKahanGroups + lane + 32 * r];
          pair_add(hi, lo, v.x, -v.y);
        }
#pragma unroll
        for (int h = 16; h >= 1; h >>= 1) {
          const float bh = __shfl_down_sync(0xffffffffu, hi, h);
          const float bl = __shfl_down_sync(0xffffffffu, lo, h);
          pair_add(hi, lo, bh, bl);
        }
        if (lane == 0) {
          reinterpret_cast<float2*>(p.rows)[((size_t)(k & 1) * G + blockIdx.x) * kNQ + warp] =
              make_float2(hi, lo);
          fence_proxy_async_global();   // the rows are read back by bulk copies
        }
      }
    }
    // the reduction scratch is overwritten by the rows' bulk copy below
    fence_proxy_async();
    if (!grid_barrier(p.bar, p.bar_base + (unsigned long long)(k + 1) * G + p.bar_extra,
                      p.wait_limit))
      s_bad = 1;
    // while thread 0 waits for the other blocks, warp 14 forms what the scalar
    // chain needs that does not depend on the sums: this stage's SumCoef and
    // the next stage's PreCoef (it starts from a = k.a, h_prev = k.h)
    if (warp == kPWarps - 2 && lane == 0) {
      s_sc = sum_coef<MODEL, PREC>(sctxv[cb], d);
      if (k < KL) {
        const int mn = k + 1 < K ? MODE_SWEEP : MODE_FLUSH;
        const int sn = sbv[cb].stage + 1 < d.nstages ? sbv[cb].stage + 1 : 0;
        const Coef& kc = sctxv[cb].k;   // of a sweep: a flush is the last pass
        const double hn = stage_step(d, sn, kc.deta, mn);
        s_qn = prestage_a(kc.a, kc.ia, kc.h, hn, d, mn, d.physical ? kc.deta : d.dt,
                          d.physical && sn == 0, d.w[sn]);
      }
    }
    __syncthreads();
    // @released
    if (s_bad) { fault = true; break; }

    // ---- after the barrier, on disjoint warps:
    //   warps 0..nl-1 fold every block's row (in block order, identically in
    //     every block); the next stage's copies wait until these latency-
    //     critical loads have landed (named barrier 1), so that they are not
    //     queued behind the copies;
    //   warps 15, 14, ... (PRE of them) issue the next stage's first LEAD
    //     planes, every PRE-th plane each (its buffers are known: a sweep
    //     swaps phi and pi, a flush swaps phi) ----
    const int ib_next = ib ^ (mode == MODE_SWEEP ? 3 : 1);
    const bool pre = k < KL;
    constexpr int kPreThreads = (1 + PRE) * 32;
    using FT = typename std::conditional<PREC != PREC_SPLIT, double, float2>::type;
    // every block's row arrives by one bulk copy into the (now free) reduction
    // scratch: one request stream per block instead of 8-byte loads of the
    // same lines by every block
    FT* srows = reinterpret_cast<FT*>(PREC != PREC_SPLIT ? (void*)sm.red : (void*)sm.kahan);
    if (warp == 0) {
      if (lane == 0) {
        const uint32_t bytes = (uint32_t)(G * kNQ * sizeof(FT));
        mbar_expect_tx(&foldbar, bytes);
        bulk_load(srows, reinterpret_cast<const FT*>(p.rows) + (size_t)(k & 1) * G * kNQ, bytes,
                  &foldbar);
        s_fold = (int)(k & 1);
      }
      __syncwarp();
      if (pre && !PLAIN) named_arrive(1, kPreThreads);   // the next stage's copies queue behind it
    }
    if constexpr (PLAIN) {   // every thread's own copies; the folding warps' after their fold
      if (pre && warp > nl) plain_prefetch<MODEL, NQ, H>(p.g.n, sm, ib_next, gq);
    }
    if (warp < nl) {
      if (!mbar_wait(&foldbar, (uint32_t)(k & 1), p.wait_limit)) atomicOr(&s_bad, 1);
      if constexpr (PREC != PREC_SPLIT) {
        double v = 0.0;
        for (int r = lane; r < G; r += 32) v += srows[(size_t)r * kNQ + slot];   // row order
#pragma unroll
        for (int h = 16; h >= 1; h >>= 1) v += __shfl_down_sync(0xffffffffu, v, h);
        if (lane == 0) sums[slot] = v;
      } else {
        float hi = 0.f, lo = 0.f;
        for (int r = lane; r < G; r += 32) {
          const float2 x = srows[(size_t)r * kNQ + slot];
          pair_add(hi, lo, x.x, x.y);
        }
#pragma unroll
        for (int h = 16; h >= 1; h >>= 1) {
          const float bh = __shfl_down_sync(0xffffffffu, hi, h);
          const float bl = __shfl_down_sync(0xffffffffu, lo, h);
          pair_add(hi, lo, bh, bl);
        }
        if (lane == 0) sums[slot] = (double)hi + (double)lo;
      }
      // @sums-written
    } else if (PREC == PREC_FP64 && warp == nl) {
      // the lattice's largest |phi| and |pi| of each field
      if (!mbar_wait(&foldbar, (uint32_t)(k & 1), p.wait_limit)) atomicOr(&s_bad, 1);
      uint32_t m[2 * NF];
#pragma unroll
      for (int i = 0; i < 2 * NF; ++i) m[i] = 0u;
      for (int r = lane; r < G; r += 32)
#pragma unroll
        for (int f = 0; f < NF; ++f) {
          const uint2 x = reinterpret_cast<const uint2*>(srows)[(size_t)r * kNQ + kNQ - kMaxFields + f];
          m[2 * f] = max(m[2 * f], x.x);
          m[2 * f + 1] = max(m[2 * f + 1], x.y);
        }
#pragma unroll
      for (int i = 0; i < 2 * NF; ++i) {
        m[i] = __reduce_max_sync(0xffffffffu, m[i]);
        if (lane == 0) s_amax[i] = 0x80000000u | m[i];
      }
    } else {
      const int l0 = kPWarps - 1 - warp;
      if (!PLAIN && pre && l0 < PRE) {
        named_sync(1, kPreThreads);
        if constexpr (!PLAIN) {
          for (int l = l0; l < LEAD; l += PRE)
            prefetch_plane<PREC, NF, VX, CORNERS, NSLOT, H>(p, sm, ib_next, gq, l);
        }
      }
      // @prefetch-issued
    }
    __syncthreads();
    // @folded
    if (tid == 0 && !s_bad) s_fold = -1;   // every folding warp saw the copy land
    if constexpr (PLAIN) {
      if (pre && warp <= nl) plain_prefetch<MODEL, NQ, H>(p.g.n, sm, ib_next, gq);
    }
    // ---- in parallel, on warps of different schedulers, identically in
    //      every block: the next stage's coefficients (warp 14: sums -> p_a
    //      kick -> scalar half-steps -> split background), the split form's
    //      re-centring (warp 12, joined to warp 14 by named barrier 2) and the
    //      bookkeeping of this stage (warp 13) ----
    // (the current Ctx is read from shared memory here, not from the sweep's
    // register copy, so that the copy's live range ends with the sweep)
    const C& cc = sctxv[cb];
    if (warp == kPWarps - 2) {
      if (pre) {
        const int mn = k + 1 < K ? MODE_SWEEP : MODE_FLUSH;
        C& nx = sctxv[cb ^ 1];
        if (lane == 0) {
          nx.set_coef(chain_coef<MODEL, PREC>(cc, s_sc, s_qn, d, sums, mn), d, mn, cc.pk);
          if constexpr (PREC == PREC_FP64) {   // the next stage's input is this stage's output
#pragma unroll
            for (int f = 0; f < NF; ++f)
              nx.shiftK[f] = (mn == MODE_FLUSH) ? flush_shift(d, ib_next, f, nx.k.c) : 0.0;
            nx.set_qref(d, ib_next);
            nx.set_fix(s_amax, fix_headroom<STENCIL>());
          }
        }
        if constexpr (PREC != PREC_FP64) {
          __syncwarp();
          named_sync(2, 64);
          if (lane == 0) nx.split_tail(d, mn, s_p0);
        }
      }
      // @chain-done
    } else if (warp == kPWarps - 4) {
      if constexpr (PREC != PREC_FP64) {
        if (pre) {
          if (lane == 0) {
            double mphi[NF], mpi[NF];
            chain_means<PREC>(cc, d, sums, mphi, mpi);
            sctxv[cb ^ 1].recenter(mphi, mpi, cc.phi0s, cc.pi0s, s_p0);
          }
          __syncwarp();
          named_arrive(2, 64);
        }
      }
    } else if (tid == kPThreads - 96) {
      post_stage<MODEL, PREC>(cc, s_sc, d, mode, sums, sbv[cb], sbv[cb ^ 1]);
      if constexpr (PREC == PREC_FP64) {
#pragma unroll
        for (int i = 0; i < 2 * NF; ++i) sbv[cb ^ 1].amax[i] = s_amax[i];
      }
      // @book-done
    }
    __syncthreads();
    // @coefficients
    cb ^= 1;
    if (s_bad) { fault = true; break; }
    if (sbv[cb].error) break;   // identical sums in every block: every block stops here
    ib = ib_next;
  }

  // copies issued for a stage that will not run (a stop after a non-finite
  // sum, or a fault) must land before the block exits (bounded waits)
  if constexpr (PLAIN) cp_async_wait<0>();
  __syncthreads();
  if (tid == 0) {
    if (fault) atomicOr(p.fault, 1);
    for (int s = 0; s < NSLOT; ++s)
      if (s_issued[s]) mbar_wait(&full[s], ((s_issued[s] - 1u) / NSLOT) & 1u);
    if (s_fold >= 0) mbar_wait(&foldbar, (uint32_t)s_fold);   // a rows copy still in flight
  }
  if (fault) return;   // the state is not trusted any more (the host poisons the simulation)
  if (blockIdx.x == 0 && tid < (int)(sizeof(Background) / 8))
    reinterpret_cast<unsigned long long*>(p.bg)[tid] =
        reinterpret_cast<const unsigned long long*>(&sbv[cb])[tid];
}

// Launch helper (one translation unit per precision and set: WIDE = the
// 13-point stencil, PLAIN = the plain staging with every stencil).  grid == 0: only set
// the kernel's shared-memory attribute and report its occupancy in *bps.
template <int PREC, bool WIDE = false, bool PLAIN = false>
cudaError_t launch_persist_impl(int model, int stencil, int vx, const PParams& p, int grid,
                                cudaStream_t s, int* bps) {
#define PYCOOL_P(M, ST, V)                                                                  \
  if constexpr (V * Pot<M>::NF * prec_word(PREC) <= 16) {                                  \
    if (model == M && stencil == ST && vx == V) {                                           \
      constexpr size_t smem =                                                               \
          RingOf<PREC, Pot<M>::NF, V, Slots<Pot<M>::NF, PREC>::NQ, halo_of<ST>()>::type::SMEM_BYTES; \
      auto kern = evolve_persist<M, ST, PREC, V>;                                           \
      if (grid == 0) {                                                                      \
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                             (int)smem);                                    \
        if (e != cudaSuccess) return e;                                                     \
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, kern, kPThreads, smem);   \
      }                                                                                     \
      cudaLaunchConfig_t cfg = {};                                                          \
      cfg.gridDim = dim3(grid);                                                             \
      cfg.blockDim = dim3(kPThreads);                                                       \
      cfg.dynamicSmemBytes = smem;                                                          \
      cfg.stream = s;                                                                       \
      cudaLaunchAttribute attr[1];                                                          \
      attr[0].id = cudaLaunchAttributeCooperative;                                          \
      attr[0].val.cooperative = 1;                                                          \
      cfg.attrs = attr;                                                                     \
      cfg.numAttrs = 1;                                                                     \
      return cudaLaunchKernelEx(&cfg, kern, p);                                             \
    }                                                                                       \
  }
#define PYCOOL_PM(X, V)                                                                     \
  X(M_FREE, 7, V) X(M_FREE, 27, V) X(M_CHAOTIC2, 7, V) X(M_CHAOTIC2, 27, V)                 \
  X(M_OSCILLON, 7, V) X(M_OSCILLON, 27, V) X(M_QBALL, 7, V) X(M_QBALL, 27, V)
#define PYCOOL_PW(X, V) X(M_FREE, 13, V) X(M_CHAOTIC2, 13, V) X(M_OSCILLON, 13, V) X(M_QBALL, 13, V)
  if constexpr (PLAIN) {
    PYCOOL_PM(PYCOOL_P, 0)
    PYCOOL_PW(PYCOOL_P, 0)
  } else if constexpr (WIDE) {
    static_assert(PREC != PREC_SPLIT, "the 13-point stencil: FP64 and split-DD");
    PYCOOL_PW(PYCOOL_P, 1)
    PYCOOL_PW(PYCOOL_P, 2)
  } else {
    PYCOOL_PM(PYCOOL_P, 1)
    PYCOOL_PM(PYCOOL_P, 2)
    if constexpr (PREC == PREC_SPLIT) { PYCOOL_PM(PYCOOL_P, 4) }
  }
#undef PYCOOL_PW
#undef PYCOOL_PM
#undef PYCOOL_P
  return cudaErrorInvalidValue;
}

}  // namespace pycool
