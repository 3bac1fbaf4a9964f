// Staging of the FP64 form's persistent kernel without TMA: any lattice side (a
// TMA box wants rows that are multiples of 16 bytes and tiles of whole boxes).
//
// A tile is w x h sites (w h <= 512, chosen by plain_tiles so that as few tiles
// as possible cover the lattice: tiles differ in w and h by at most one, and no
// thread row is tied to a lattice row), one site per thread.  Each thread
// copies its own site's values of the planes ahead, and at most one cell of the
// tile's halo ring (periodic indices), with 8-byte cp.async into its own
// places of a shared-memory ring; it alone reads them again, so a copy needs no
// barrier, only the thread's own cp.async group count.  The thread drifts its
// cells of plane g + 1 into one of four drift buffers (fixed point or float64),
// its warp arrives on the buffer's mbarrier, and after the wait for plane g it
// sums the stencil of plane g from shared memory and puts out the plane H below,
// whose drifted field and momentum it still holds in the ring.  As in the other
// stages there is no block barrier in the z loop.
//
// Bound by the float64 pipe.  Measured on GB300, per stage, against the
// per-stage kernels (sweep_plain, sweep_wide: ragged 32 x 8 tiles in two uneven
// waves of blocks, float64 stencils, a launch per stage): chaotic 16^3 24.4 ->
// 8.5 us, 37^3 27.5 -> 9.8, 100^3 144 -> 44, with 27 points 209 -> 47, with 13
// points 238 -> 48, oscillon 203^3 435 -> 201.  The split-FP32 form keeps the
// per-stage kernels at these sides: it was faster here too (100^3 40 -> 18 us),
// but its float32 sums in another order moved the field by up to 4e-9 of itself
// where a one-field background passes near zero (Ctx::recenter).
#pragma once

#include "persist.cuh"

namespace pycool {

constexpr int kPlainHalo = 256;                       // halo cells of a tile at most
constexpr int kPlainCells = kPThreads + kPlainHalo;   // cells of a tile with its halo

// Shared memory: own[OSLOT][NF][phi, pi][512], halo[HSLOT][NF][phi, pi][256]
// and the drift buffers fx[NDRIFT][NF][768].  LEAD planes of copies are in
// flight ahead of the plane being drifted; an own slot is needed until the
// plane has been put out, H + 1 planes after its drift.
template <int NF, int NQ, int H>
struct PlainRing {
  static constexpr int OSLOT = 6;
  static constexpr int LEAD = OSLOT - H - 2;
  static constexpr int HSLOT = LEAD + 1;
  static constexpr int NDRIFT = 4;
  static constexpr int NSLOT = 1;   // no TMA ring
  static constexpr int FOLD = NQ + 1;
  static constexpr int PRE = 1;
  static constexpr int OWN = NF * 2 * kPThreads, HALO = NF * 2 * kPlainHalo;
  static constexpr int FX = NF * kPlainCells;
  static constexpr int HALO_OFF = OSLOT * OWN, FX_OFF = HALO_OFF + HSLOT * HALO;
  static constexpr int RING_BYTES = (FX_OFF + NDRIFT * FX) * 8;
  static constexpr int DRIFT_WORDS = 0;
  static constexpr int SMEM_BYTES = RING_BYTES + NQ * kPThreads * 8;
  static_assert(SMEM_BYTES <= kPSmemBudget, "shared memory of the persistent kernel");
  static_assert(RING_BYTES % 16 == 0, "the rows' bulk copy lands behind the ring");
};

// An 8-byte asynchronous copy into the thread's own place (dst: a shared
// address, OFF bytes behind it an instruction's immediate).
template <int OFF> __device__ __forceinline__ void cp_async_word(uint32_t dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0+%2], [%1], 8;" ::"r"(dst), "l"(src), "n"(OFF)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// A thread's cells of a unit (x0 | w << 16, y0 | h << 16, z0, planes): in-plane
// offsets in the lattice (own, halo; -1: none) and in a drift buffer whose rows
// are rs = w + 2 H cells.
struct PlainCells {
  int own, ownc, halo, haloc, rs;
};
template <int H>
__device__ __forceinline__ PlainCells plain_cells(int4 u, int n) {
  PlainCells c;
  const int x0 = u.x & 0xffff, w = u.x >> 16, y0 = u.y & 0xffff, h = u.y >> 16;
  const int t = threadIdx.x;
  c.rs = w + 2 * H;
  c.own = c.halo = -1;
  c.ownc = H * c.rs + H;   // a thread without a site reads the first one's neighbours
  c.haloc = 0;
  if (t < w * h) {
    const int ly = t / w, lx = t - ly * w;
    c.own = (y0 + ly) * n + x0 + lx;
    c.ownc = (ly + H) * c.rs + lx + H;
  }
  if (t < 2 * H * (c.rs + h)) {   // 2H full rows, then 2H cells beside each of the h rows
    int row, col;
    if (t < 2 * H * c.rs) {
      const int r = t / c.rs;
      col = t - r * c.rs;
      row = r < H ? r : h + r;
    } else {
      const int t2 = t - 2 * H * c.rs, k = t2 % (2 * H);
      row = t2 / (2 * H) + H;
      col = k < H ? k : w + k;
    }
    c.halo = wrapi(y0 - H + row, n) * n + wrapi(x0 - H + col, n);
    c.haloc = row * c.rs + col;
  }
  return c;
}

// A position in the block's planes: the thread's cells there and the plane's own
// and halo slots in the ring (elements).  The plane loop is a chain that each warp
// walks with few others beside it (16 on the SM), so its instructions count: plane
// offsets are 32-bit element indices (N_f n^3 < 2^32), advanced instead of
// multiplied, and so are the slots.
template <int H, typename RG>
struct PlainPos {
  int ui, left;      // unit, planes of it to come (0: past the last unit)
  uint32_t zo;       // n^2 z of the plane
  uint32_t os, hs;
  PlainCells c;
  __device__ __forceinline__ void enter(const PShared& sm, int n) {
    left = 0;
    if (ui < sm.nunits) {
      const int4 u = sm.units[ui];
      c = plain_cells<H>(u, n);
      left = u.w;
      zo = (uint32_t)wrapi(u.z - H, n) * (uint32_t)(n * n);
    }
  }
  // the block's first plane, ring plane gq
  __device__ __forceinline__ void start(const PShared& sm, int n, uint32_t gq) {
    ui = 0;
    zo = 0u;
    os = (gq % RG::OSLOT) * RG::OWN;
    hs = (gq % RG::HSLOT) * RG::HALO;
    enter(sm, n);
  }
  __device__ __forceinline__ bool in() const { return left > 0; }
  __device__ __forceinline__ void next(const PShared& sm, int n, uint32_t nn, uint32_t S) {
    os = os == (RG::OSLOT - 1) * RG::OWN ? 0u : os + RG::OWN;
    hs = hs == (RG::HSLOT - 1) * RG::HALO ? 0u : hs + RG::HALO;
    zo += nn;
    if (zo == S) zo = 0u;
    if (--left == 0) {
      ++ui;
      enter(sm, n);
    }
  }
};
// slot s (elements) of a ring of N slots of E elements, K further on
template <int N, int E, int K> __device__ __forceinline__ uint32_t ring_slot(uint32_t s) {
  static_assert(K >= 0 && K < N, "one wrap");
  return s >= (uint32_t)((N - K) * E) ? s - (uint32_t)((N - K) * E) : s + (uint32_t)(K * E);
}

// A potential given at run time: its stage (rt_kick) finds the field drifted
// (SimDesc::rt_phis) and V' and V at every site in arrays.
template <int MODEL> constexpr bool runtime_pot() {
  return MODEL == M_RUNTIME1 || MODEL == M_RUNTIME2;
}

// Copies of the plane at `pos` into slots os, hs of the ring and one commit, always: the
// groups a thread has committed count the planes.
template <int MODEL, int NQ, int H, typename Pos>
__device__ __forceinline__ void plain_issue(int n, uint32_t nn, uint32_t S, const PShared& sm,
                                            Pos& pos, int ib, uint32_t os, uint32_t hs) {
  constexpr bool RT = runtime_pot<MODEL>();
  constexpr int NF = Pot<MODEL>::NF;
  using T = double;
  using RG = PlainRing<NF, NQ, H>;
  constexpr int W = sizeof(T);
  if (pos.in()) {
    const SimDesc& d = *sm.d;
    const T* phi = RT ? (const T*)d.rt_phis : (const T*)d.phi[ib & 1];
    const T* pi = (const T*)d.pi[(ib >> 1) & 1];
    const uint32_t ring = smem_u32(sm.ring) + threadIdx.x * W;
    const uint32_t own = ring + os * W, hal = ring + hs * W;
    constexpr int HB = RG::HALO_OFF * W;
    if (pos.c.own >= 0) {
      const uint32_t o = pos.zo + (uint32_t)pos.c.own;
      cp_async_word<0>(own, phi + o);
      cp_async_word<kPThreads * W>(own, pi + o);
      if constexpr (NF == 2) {
        cp_async_word<2 * kPThreads * W>(own, phi + (o + S));
        cp_async_word<3 * kPThreads * W>(own, pi + (o + S));
      }
    }
    if (pos.c.halo >= 0) {
      const uint32_t o = pos.zo + (uint32_t)pos.c.halo;
      cp_async_word<HB>(hal, phi + o);
      if constexpr (!RT) cp_async_word<HB + kPlainHalo * W>(hal, pi + o);
      if constexpr (NF == 2) {
        cp_async_word<HB + 2 * kPlainHalo * W>(hal, phi + (o + S));
        if constexpr (!RT) cp_async_word<HB + 3 * kPlainHalo * W>(hal, pi + (o + S));
      }
    }
    pos.next(sm, n, nn, S);
  }
  cp_async_commit();
}

// The first LEAD planes of a stage (every thread of the block).
template <int MODEL, int NQ, int H>
__device__ __forceinline__ void plain_prefetch(int n, const PShared& sm, int ib, uint32_t gq) {
  using RG = PlainRing<Pot<MODEL>::NF, NQ, H>;
  const uint32_t nn = (uint32_t)(n * n), S = nn * (uint32_t)n;
  PlainPos<H, RG> pos;
  pos.start(sm, n, gq);
  for (int l = 0; l < RG::LEAD; ++l)
    plain_issue<MODEL, NQ, H>(n, nn, S, sm, pos, ib, pos.os, pos.hs);
}

// One stage over this block's units (see the head of this file); the sums go to
// accd.
template <int MODEL, int STENCIL, int MODE, bool FIX>
__device__ __forceinline__ bool stage_plain(int n, const Ctx<MODEL, PREC_FP64>& cx0, const PShared& sm,
                                            uint32_t gq, int ib, double* accd,
                                            HiMax<Pot<MODEL>::NF>& hm) {
  constexpr bool RT = runtime_pot<MODEL>();
  using C = Ctx<MODEL, PREC_FP64>;
  using T = double;
  using E = typename FixElem<FIX>::type;
  using SL = typename C::SL;
  constexpr int NF = C::NF, NQ = SL::NQ, H = halo_of<STENCIL>();
  constexpr bool CORNERS = StencilW<STENCIL>::kCorners;
  constexpr bool WIDE = STENCIL == 13;
  using RG = PlainRing<NF, NQ, H>;
  constexpr int NB = RG::NDRIFT, LEAD = RG::LEAD;
  const SimDesc& d = *sm.d;
  const int tid = threadIdx.x, lane = tid & 31;
  const uint32_t nn = (uint32_t)(n * n), S = nn * (uint32_t)n;
  T* __restrict__ phi_out = (T*)d.phi[(ib & 1) ^ 1];
  T* __restrict__ pi_out = (T*)d.pi[((ib >> 1) & 1) ^ 1];
  T* const own = (T*)sm.ring + tid;
  const T* const hal = (const T*)sm.ring + RG::HALO_OFF + tid;
  E* const fxb = (E*)((T*)sm.ring + RG::FX_OFF);
  // integer sums (13 points: float64 sums too) are D times the weights' common
  // denominator, which goes into the kick's coefficient and, after the stage,
  // into sum phi D
  constexpr bool TIMES = WIDE || (FIX && STENCIL == 27);
  C cx = cx0;
  if constexpr (TIMES) cx.kD *= 1.0 / fix_weight<STENCIL>();
  const E w1 = (E)16, w2 = (E)0 - (E)1, w0 = (E)0 - (E)90;   // 13 points, times 12
  bool ok = true;

  // Three positions run through the planes: copied, drifted, put out.  Where
  // registers are short (two fields: the Q-ball spilled, 3 to 6 % slower) only
  // the last one keeps its slots and cells, and the others' are derived from them.
  constexpr bool RUN = NF == 1;
  PlainPos<H, RG> ip, dp;   // next plane to copy, next plane to drift
  ip.start(sm, n, gq);
  for (int l = 0; l < LEAD && ip.in(); ++l) ip.next(sm, n, nn, S);
  if constexpr (RUN) dp.start(sm, n, gq);
  // own slot of plane g - H and halo slot of plane g; here for g = gq - 1
  uint32_t os = ((gq + RG::OSLOT - 1 - H) % RG::OSLOT) * RG::OWN;
  uint32_t hs = ((gq + RG::HSLOT - 1) % RG::HSLOT) * RG::HALO;
  auto advance = [&]() {
    os = os == (RG::OSLOT - 1) * RG::OWN ? 0u : os + RG::OWN;
    if constexpr (!RUN) hs = hs == (RG::HSLOT - 1) * RG::HALO ? 0u : hs + RG::HALO;
  };
  // the copies of plane g + 1 + LEAD
  static_assert(RG::OSLOT == LEAD + H + 2 && RG::HSLOT == LEAD + 1, "slots of the planes ahead");
  auto issue = [&]() {
    if constexpr (RUN)
      plain_issue<MODEL, NQ, H>(n, nn, S, sm, ip, ib, ip.os, ip.hs);
    else
      plain_issue<MODEL, NQ, H>(n, nn, S, sm, ip, ib,
                                ring_slot<RG::OSLOT, RG::OWN, RG::OSLOT - 1>(os), hs);
  };
  // drift of plane gg = g + 1 with the thread's cells there: own cell in place and
  // into the drift buffer, the halo cell into the drift buffer
  auto drift = [&](uint32_t gg, const PlainCells& dc) {
    T* o = own + (RUN ? dp.os : ring_slot<RG::OSLOT, RG::OWN, H + 1>(os));
    const T* h = hal + (RUN ? dp.hs : ring_slot<RG::HSLOT, RG::HALO, 1>(hs));
    E* fx = fxb + (gg % NB) * RG::FX;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      const int ex = cx.fx[f];
      if (dc.own >= 0) {
        T a = o[f * 2 * kPThreads];
        if constexpr (!RT) {
          a = madd(cx.cdrift, o[(f * 2 + 1) * kPThreads], a);
          o[f * 2 * kPThreads] = a;
        }
        fx[f * kPlainCells + dc.ownc] = fix_in(a, ex, (E*)nullptr);
      }
      if (dc.halo >= 0) {
        T a = h[f * 2 * kPlainHalo];
        if constexpr (!RT) a = madd(cx.cdrift, h[(f * 2 + 1) * kPlainHalo], a);
        fx[f * kPlainCells + dc.haloc] = fix_in(a, ex, (E*)nullptr);
      }
    }
    __syncwarp();   // the lanes' writes before lane 0's arrival (release)
    if (lane == 0) mbar_arrive(&sm.dbar[gg % NB]);
  };

  uint32_t g = gq;
  PlainCells c;   // the thread's cells of the plane put out
  constexpr bool KEEP = !RUN && MODEL != M_QBALL;   // (the Q-ball forms them again: registers)
  if (sm.nunits > 0) {
    if constexpr (!RUN) c = plain_cells<H>(sm.units[0], n);
    issue();
    cp_async_wait<LEAD>();
    if constexpr (RUN) {
      drift(g, dp.c);
      dp.next(sm, n, nn, S);
    } else {
      drift(g, c);
    }
  }
  advance();
  for (int i = 0; i < sm.nunits && ok; ++i) {
    const int4 u = sm.units[i];
    const int Q = u.w;
    if (!KEEP || i > 0) c = plain_cells<H>(u, n);
    const bool valid = c.own >= 0;
    // 7- and 27-point: part_m, so_m as in stage_fp64; 13-point: the z queue of stage_fp64_wide
    E qa[NF], qb[NF], qc[NF], qd[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) qa[f] = qb[f] = qc[f] = qd[f] = (E)0;
    uint32_t oz = (uint32_t)u.z * nn + (uint32_t)c.own;   // the next output
    for (int q = 0; q < Q; ++q, ++g, advance()) {
      issue();
      if constexpr (RUN) {
        if (dp.in()) {
          cp_async_wait<LEAD>();
          drift(g + 1, dp.c);
          dp.next(sm, n, nn, S);
        }
      } else {
        PlainCells dc = c;   // the next plane may be the next unit's first
        if (q + 1 == Q && i + 1 < sm.nunits) dc = plain_cells<H>(sm.units[i + 1], n);
        if (q + 1 < Q || i + 1 < sm.nunits) {
          cp_async_wait<LEAD>();
          drift(g + 1, dc);
        }
      }
      double rv[RT ? NF + 1 : 1];   // run-time potential: V' and V of the plane put out
      if constexpr (RT) {
        const bool put = valid && q >= 2 * H;
#pragma unroll
        for (int f = 0; f < NF; ++f)
          rv[f] = put && MODE == MODE_SWEEP ? __ldcg(d.rt_dV + (oz + f * S)) : 0.0;
        rv[NF] = put ? __ldcg(d.rt_V + oz) : 0.0;
      }
      // every warp has drifted plane g
      ok = mbar_wait(&sm.dbar[g % NB], (g / NB) & 1, sm.limit);
      if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
      const bool mid = q >= H && q < Q - H;   // a plane whose sites are output
      E D[NF];
#pragma unroll
      for (int f = 0; f < NF; ++f) {
        const E* fx = fxb + (g % NB) * RG::FX + f * kPlainCells + c.ownc;
        const int rs = c.rs;
        const E ctr = fx[0];
        if constexpr (WIDE) {
          E m = (E)0;
          if (mid) {
            const E nr = (fx[-rs] + fx[rs]) + (fx[-1] + fx[1]);
            const E fr = (fx[-2 * rs] + fx[2 * rs]) + (fx[-2] + fx[2]);
            m = fix_mad(w0, ctr, fix_mad(w2, fr, w1 * nr));
          }
          D[f] = fix_mad(w2, ctr, qb[f]);   // plane p - 2: its last term
          const E np1 = fix_mad(w1, ctr, qa[f]);
          qa[f] = fix_mad(w2, qd[f], fix_mad(w1, qc[f], m));
          qb[f] = np1;
          qd[f] = qc[f];
          qc[f] = ctr;
        } else {
          E smid = ctr, so = ctr;
          if (CORNERS || mid) {
            const E faces = (fx[-rs] + fx[rs]) + (fx[-1] + fx[1]);
            if constexpr (CORNERS)
              fix_parts27(ctr, faces, (fx[-rs - 1] + fx[-rs + 1]) + (fx[rs - 1] + fx[rs + 1]),
                          smid, so);
            else
              smid = fix_mid7(ctr, faces);
          }
          D[f] = qa[f] + so;
          if (mid) qa[f] = qb[f] + smid;
          qb[f] = so;
        }
      }
      if (q >= 2 * H) {  // output plane z0 + q - 2 H
        if (valid) {
          T phj[NF], Dj[NF], pmj[NF], pnj[NF];
          const T* r = own + os;
#pragma unroll
          for (int f = 0; f < NF; ++f) {
            phj[f] = r[f * 2 * kPThreads];
            pmj[f] = r[(f * 2 + 1) * kPThreads];
            Dj[f] = fix_out(D[f], cx.fx[f]);
          }
          if constexpr (RT) {
#pragma unroll
            for (int f = 0; f < NF; ++f) {
              if (MODE == MODE_SWEEP) {
                pnj[f] = madd(cx.kD, Dj[f], madd(-cx.kV, rv[f], pmj[f]));
                accd[SL::PI2] = madd(pnj[f], pnj[f], accd[SL::PI2]);
                accd[SL::PHID] = madd(phj[f], Dj[f], accd[SL::PHID]);
              } else {
                pnj[f] = pmj[f];
                accd[SL::PI2 + f] = madd(pmj[f], pmj[f], accd[SL::PI2 + f]);
                accd[SL::PHID + f] = madd(phj[f], Dj[f], accd[SL::PHID + f]);
                const T dd = phj[f] - cx.shiftK[f];
                accd[SL::DPHI + f] += dd;
                accd[SL::DPHI2 + f] = madd(dd, dd, accd[SL::DPHI2 + f]);
              }
            }
            accd[SL::V] += rv[NF];
          } else {
            cx.site(MODE, phj, Dj, pmj, pnj, accd);
          }
#pragma unroll
          for (int f = 0; f < NF; ++f) {
            hm.add(2 * f, phj[f]);
            hm.add(2 * f + 1, pnj[f]);
            __stwb(phi_out + (oz + f * S), phj[f]);
            if (MODE == MODE_SWEEP) __stwb(pi_out + (oz + f * S), pnj[f]);
          }
        }
        oz += nn;
      }
    }
  }
  if constexpr (TIMES) {
#pragma unroll
    for (int f = 0; f < NF; ++f) accd[SL::PHID + f] *= 1.0 / fix_weight<STENCIL>();
  }
  return ok;
}

}  // namespace pycool
