// SIGMAKIN with helicity-shared currents (the default kernel of both modes).
//
// Same result as the straight-line kernel (sigmakin.cuh) — the same Feynman
// diagrams, colour flows and colour matrix (Sec. 2) — organised for GB300:
//   * an off-shell current over legs S depends only on the helicities of S,
//     so each current is computed once per event for each of its 2^|S|
//     helicity variants (not once per event helicity), into shared memory;
//   * every diagram's amplitude is a contraction sum_i X_i Y_i of two such
//     objects, so that a helicity pays only the contractions.  gg -> t t~ g and
//     gg -> t t~ g g run the ordered program (gen/procgen.py): colour-ordered
//     currents summed over their diagrams before they are contracted, 12 and 55
//     contractions per helicity for 18 and 159 amplitude terms; the smaller
//     processes contract diagram by diagram;
//   * currents and operands are item tables walked by short loops (lanes take
//     one item for each of the CTA's units); the contractions are generated
//     straight-line code.
// The mixed mode takes pairs of events: a lane value is an f2, one event per
// half, and every FP32 operation one paired instruction (mg_types.cuh).
// CTA of NT threads = units (pairs of events in the mixed mode) x ngood
// helicities.  Phases:
//   1. per-event momenta, momentum sums and propagator factors, external
//      wavefunctions;
//   2. current variants, level by level (a level only reads earlier levels);
//   3. the contractions' operands (all threads), then one thread per (unit,
//      helicity) contracts them into its colour flows J (registers);
//   4. colour sum (CUDA cores, or tcgen05 as in sigmakin.cuh) and the
//      fixed-order FP64 helicity sum.
// What bounds it (gg -> t t~ g g mixed, 2^20 events): the bytes that the
// contractions load from shared memory into registers (128 per clock and SM; with
// the items' loads 60 % of the kernel's cycles) and the latency of dependent FMAs
// at 8 warps per SM (FMA pipe 49 % busy): 9.8 ms, against 18.0 ms for the
// diagram-wise program on single events.  In FP64 the FP64 pipe (90 % busy for gg -> t t~ g).
#pragma once
#include <type_traits>

#include "dfl.cuh"
#include "rambo.cuh"
#include "rng.cuh"
#include "sigmakin.cuh"

namespace mg {

// threads per CTA of the mixed kernels of six and more colour flows, and their
// CTAs per SM (six flows; more: one).  Measured on pairs of events: gg -> t t~ g g,
// 2^20 events, one CTA of 256 threads 10.3 ms, two of 128 11.5 ms, three of 128
// (168 registers, spills) 11.1 ms; gg -> t t~ g, 262147 events, two of 256 540 us,
// three of 128 612 us.
#ifndef MG_HS_NT
#define MG_HS_NT 256
#endif
#ifndef MG_HS_CTAS
#define MG_HS_CTAS 2
#endif

// current slots and contraction operands in shared memory: the ordered
// program's are planar
template <class P, class R, int N>
using HsSlots = std::conditional_t<P::HS_ORDERED, PlanarSlots<R, N>, Slots<R, N>>;

// Lane type of a kernel: pairs of events (f2) in the mixed mode with the
// CUDA-core colour sum; the tensor-core colour sum takes one row per thread, and
// the one-flow process is mostly wavefunctions and tables (2^19 events: single
// 214 us, pairs 272 us; gg -> t t~, 2^20 events: 781 and 630 us).
template <class P, class R, int CS>
using HsLane = std::conditional_t<std::is_same_v<R, float> && CS == CS_SIMT && (P::NCOLOR > 1), f2, R>;

// CTA shape.  A thread takes one helicity of one unit, a unit being the events
// of a lane (a pair in the mixed mode).  FUSED: the kernel with RAMBO inside.
template <class P, class R, int CS = CS_SIMT, bool FUSED = false>
struct HsCfg {
  using V = HsLane<P, R, CS>;
  static constexpr int EW = LaneOf<V>::EW;
  // measured: 128 threads for pairs of g g -> t t~ events (2^20 events 565 us, 256
  // threads 632 us) and for FP64 e+e- -> mu+mu- (200003 events 1256 us, 1301 us);
  // 256 for FP64 g g -> t t~ (100003 events 914 us, 128 threads 974 us) and mixed
  // e+e- -> mu+mu- (200003 events 91 us, 97 us), as for the larger processes.  With
  // RAMBO inside, e+e- -> mu+mu- waits for one lane per event: CTAs of half the
  // threads, four per SM instead of two, are the faster ones (131072 events mixed
  // 115 us, 256 threads 167 us; not with the tensor-core colour sum, 346 and 320 us).
  static constexpr bool HALF = P::NCOLOR == 1 ? sizeof(R) == 8 || (FUSED && CS == CS_SIMT) : P::NCOLOR == 2 && EW == 2;
  static constexpr int NT = HALF ? 128 : EW == 2 ? MG_HS_NT : 256;
  static constexpr int EVMIN = (NT / P::NHEL) > 0 ? (NT / P::NHEL) : 1;  // units, all helicities good
  // room for groups of fewer helicities than all: four times the units with one
  // flow (four of the sixteen helicities of e+e- -> mu+mu- are good); none for the
  // others, whose shared memory then admits more CTAs per SM (2^20 g g -> t t~ events
  // in pairs 629 -> 565 us, 50021 FP64 gg -> t t~ g events 2449 -> 2226 us).  Masks of
  // few helicities leave threads idle in the contractions, a small part of these
  // processes (262144 g g -> t t~ events with 1, 4 and 16 of 16 helicities 131, 134 and
  // 133 us; with room and single events 141, 146 and 217 us)
  static constexpr int MORE = P::NCOLOR == 1 ? 4 : 1;
  static constexpr int EVWANT = (MORE * EVMIN) < 32 ? MORE * EVMIN : 32;
  // shared memory for the currents and the contractions' operands
  static constexpr int CTAS = P::NCOLOR < 6 || sizeof(R) != 4 ? 1 : EW == 2 ? (P::NCOLOR >= 24 ? 1 : MG_HS_CTAS)
                                                             : (P::NCOLOR >= 24 ? 2 : 3);
  static constexpr size_t CUR_BUDGET = 192 * 1024 / CTAS;
  static constexpr size_t EV_BYTES =
      (size_t)(P::HS_NSLOT + P::HS_XCAP) * sizeof(W4<V>) + (size_t)P::HS_NSC * sizeof(cx<V>);
  static constexpr int FIT = (int)(CUR_BUDGET / EV_BYTES);
  static constexpr int EVCAP = FIT < EVWANT ? (FIT > EVMIN ? FIT : EVMIN) : EVWANT;
  static constexpr int KP = ((P::NCOLOR + 15) / 16) * 16;
  static constexpr int NP = KP;
  static constexpr int MBLK = NT / 128;
};

template <class P, class R, int CS, bool FUSED = false>
struct HsLayout {
  using H = HsCfg<P, R, CS, FUSED>;
  using V = typename H::V;
  static constexpr int EW = H::EW;
  static constexpr int NT = H::NT, EVCAP = H::EVCAP, KP = H::KP, NP = H::NP, MBLK = H::MBLK;
  static constexpr bool TC = CS == CS_TC;
  static constexpr size_t o_proptab = 0;  // {momentum entry, line kind} per propagator
  static constexpr size_t o_md = align_up(o_proptab + 8 * P::NPROP, 16);  // momentum-entry descriptors (int4)
  static constexpr size_t o_good = align_up(o_md + 16 * P::NMOM, 16);
  static constexpr size_t o_misc = align_up(o_good + 4 * P::NHEL, 16);
  // mixed mode: {m^2 hi, m^2 lo, m w, 0} of the top and of the Z
  static constexpr size_t o_mconst = align_up(o_misc + 48, 16);
  static constexpr size_t o_p = align_up(o_mconst + 32, 16);
  // the next group's momenta (FP64), copied asynchronously while this group runs
  static constexpr size_t o_ps = align_up(o_p + 8 * EW * EVCAP * P::NPAR * 4, 16);
  static constexpr size_t o_K = align_up(o_ps + 8 * EW * EVCAP * P::NPAR * 4, 16);
  // momentum-table entries (V) from one unit to the next: an odd number of
  // 16-byte words, so that one entry of the CTA's units falls in different
  // bank groups (the lanes of a warp read it for several units at once)
  static constexpr int KEV =
      4 * P::NMOM + ((4 * P::NMOM * (int)sizeof(V) / 16) % 2 == 0 ? 16 / (int)sizeof(V) : 0);
  static constexpr size_t o_pr = align_up(o_K + sizeof(V) * EVCAP * KEV, 16);
  static constexpr size_t o_m2 = align_up(o_pr + 2 * sizeof(V) * EVCAP * P::NPROP, 16);
  // variant of a leg set for a helicity: vt[row * NHEL + ihel]
  static constexpr size_t o_vt = align_up(o_m2 + sizeof(R) * EW * NT, 16);
  static constexpr size_t o_U = align_up(o_vt + (size_t)P::HS_NVT * P::NHEL, TC ? 1024 : 128);
  // union: current variants + contraction operands (phases 2-3), then the tensor-core
  // A tiles and, after them, the colour matrix as the B operand (phase 4).
  // Per-unit strides in 16-byte words, padded so that one slot of the CTA's
  // units falls in different bank groups: the lanes of a warp take an item
  // for several units at once (the plane stride, a multiple of 8 words for
  // the processes' slot counts, would otherwise map them to one group).
  static constexpr int EVPAD = EVCAP >= 8 ? 1 : 8 / EVCAP;
  static constexpr int CUR_EV = P::HS_NSLOT * Slots<V, 1>::NPL + EVPAD;
  static constexpr int X_EV =
      P::HS_XCAP * Slots<V, 1>::NPL + (int)(align_up((size_t)P::HS_NSC * sizeof(cx<V>), 128) / 16) + EVPAD;
  static constexpr size_t o_cur = o_U;
  static constexpr size_t o_x = o_U + 16 * size_t(EVCAP) * CUR_EV;
  static constexpr size_t o_A = o_U;
  static constexpr size_t tileA = 128 * KP * 2;
  static constexpr size_t u_bytes = 16 * size_t(EVCAP) * (CUR_EV + X_EV);
  static constexpr size_t a_bytes = TC ? 3 * MBLK * tileA : 0;  // one component's three splits
  static constexpr size_t o_B = o_U + a_bytes;  // copied in for every group's colour sum
  static constexpr size_t b_bytes = TC ? size_t(NP) * KP * 2 : 0;
  static constexpr size_t bytes = o_U + (u_bytes > a_bytes + b_bytes ? u_bytes : a_bytes + b_bytes);
  static_assert(!TC || o_B % 1024 == 0, "B operand on a 1024-byte boundary");
  static constexpr uint32_t TMEM_COLS = tc::tmem_cols(MBLK * 2 * NP);
  static_assert(!TC || NT % 128 == 0, "CTA rows must fill 128-row MMA blocks");
  static_assert(TMEM_COLS <= 512, "TMEM holds 512 columns");
  static_assert(bytes <= 232448, "shared memory per CTA above the 227 KB limit");
};

// Tensor-core colour sum of the CTA's NT rows with J in registers (layout and
// three-term BF16 split as in colour_tc.cuh).  Two passes, real then imaginary
// part, so that one component's A tiles fit in the dead current-variant
// storage: Y_c = A_c B lands in TMEM columns [c NP, (c+1) NP).
template <class P, class L>
__device__ __forceinline__ float colour_sum_tc_regs(unsigned char* smem, const cx<float>* J, uint32_t tmem,
                                                    uint32_t mbar) {
  constexpr int NC = P::NCOLOR, KP = L::KP;
  const int tid = threadIdx.x;
  const int b = tid >> 7, r = tid & 127;
  bool ok = true;
  {  // the colour matrix (BF16 B operand) into the union, free from here on
    const uint4* src = reinterpret_cast<const uint4*>(P::colour_bf16_image());
    uint4* dst = reinterpret_cast<uint4*>(smem + L::o_B);
    for (int i = tid; i < (int)(L::b_bytes / 16); i += L::NT) dst[i] = src[i];
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    if (c == 1) {
      // pass 0's MMAs have read its tiles once every thread saw the barrier
      // complete; a timed-out wait ends both passes for the whole CTA
      if (__syncthreads_or(!ok)) {
        tc::mbar_wait(mbar, 0);
        return __int_as_float(0x7fc00000);
      }
    }
#pragma unroll
    for (int k0 = 0; k0 < KP; k0 += 8) {
      uint32_t w[3][4];
#pragma unroll
      for (int q = 0; q < 8; q += 2) {
        uint16_t hb[3][2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int k = k0 + q + u;
          const float x = k < NC ? (c == 0 ? J[k].re : J[k].im) : 0.0f;
          const uint16_t h = tc::bf16_bits(x);
          const float r1 = x - tc::bf16_value(h);
          const uint16_t m = tc::bf16_bits(r1);
          const uint16_t l = tc::bf16_bits(r1 - tc::bf16_value(m));
          hb[0][u] = h; hb[1][u] = m; hb[2][u] = l;
        }
#pragma unroll
        for (int sp = 0; sp < 3; ++sp) w[sp][q >> 1] = (uint32_t)hb[sp][0] | ((uint32_t)hb[sp][1] << 16);
      }
#pragma unroll
      for (int sp = 0; sp < 3; ++sp) {
        unsigned char* tile = smem + L::o_A + (sp * L::MBLK + b) * L::tileA;
        *reinterpret_cast<uint4*>(tile + tc::kmajor_offset<KP>(r, k0)) =
            make_uint4(w[sp][0], w[sp][1], w[sp][2], w[sp][3]);
      }
    }
    tc::fence_async_shared();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      constexpr uint32_t idesc = tc::idesc_bf16(128, L::NP);
      constexpr uint32_t LBO = 128, SBO = (KP / 8) * 128;
      const uint32_t bbase = tc::smem_addr(smem + L::o_B);
#pragma unroll
      for (int bb = 0; bb < L::MBLK; ++bb) {
        const uint32_t d = tmem + (uint32_t)((bb * 2 + c) * L::NP);
#pragma unroll
        for (int sp = 0; sp < 3; ++sp) {
          const uint32_t abase = tc::smem_addr(smem + L::o_A + (sp * L::MBLK + bb) * L::tileA);
#pragma unroll
          for (int j = 0; j < KP / 16; ++j)
            tc::mma_bf16(d, tc::smem_desc(abase + j * 256, LBO, SBO), tc::smem_desc(bbase + j * 256, LBO, SBO),
                         idesc, (sp | j) != 0);
        }
      }
      tc::mma_commit(mbar);
    }
    ok = tc::mbar_wait(mbar, (uint32_t)c);
  }
  tc::fence_after_sync();
  const int warp = tid >> 5;
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
  float yr[L::NP], yi[L::NP];
#pragma unroll
  for (int c0 = 0; c0 < L::NP; c0 += 16) {
    tc::tmem_ld16(tmem + lane_base + (uint32_t)((b * 2 + 0) * L::NP + c0), yr + c0);
    tc::tmem_ld16(tmem + lane_base + (uint32_t)((b * 2 + 1) * L::NP + c0), yi + c0);
  }
  tc::tmem_wait_ld();
  float s = 0.0f;
#pragma unroll
  for (int k = 0; k < NC; ++k) s += J[k].re * yr[k] + J[k].im * yi[k];
  s *= 1.0f / (float)P::CDEN;
  if (!ok) {
    tc::mbar_wait(mbar, 1);  // second bounded wait for the MMAs still in flight
    s = __int_as_float(0x7fc00000);
  }
  return s;
}

// |M_h|^2 = J^dagger C J / CDEN on CUDA cores with C real symmetric:
//   sum_i J_i^* (C_ii J_i + 2 sum_{j>i} C_ij J_j)  (real part; the imaginary parts cancel)
// — each off-diagonal entry once, half the multiply-adds of the row-wise form.
template <class P>
__host__ __device__ constexpr bool colour_matrix_symmetric() {
  for (int i = 0; i < P::NCOLOR; ++i)
    for (int j = 0; j < i; ++j)
      if (P::cnum(i, j) != P::cnum(j, i)) return false;
  return true;
}
// f(std::integral_constant<int, i>) for i = B .. E - 1: indices that are
// compile-time constants by construction (the colour matrix entries below are
// then immediates, whatever the unroller decides inside a large loop body)
template <int B, int E, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    static_for<B + 1, E>(f);
  }
}

// (a.re b.re + c.re, a.im b.im + c.im): one paired instruction in FP32
template <class R>
__device__ __forceinline__ cx<R> pair_fma(cx<R> a, cx<R> b, cx<R> c) {
  if constexpr (sizeof(R) == 4) {
    const float2 r = __ffma2_rn(make_float2(a.re, a.im), make_float2(b.re, b.im), make_float2(c.re, c.im));
    return cx<R>(r.x, r.y);
  } else {
    return cx<R>(fmac(a.re, b.re, c.re), fmac(a.im, b.im, c.im));
  }
}

template <class P, class R>
__device__ __forceinline__ R colour_sum_sym(const cx<R>* J) {
  static_assert(colour_matrix_symmetric<P>(), "colour matrix must be symmetric");
  constexpr int NC = P::NCOLOR;
  if constexpr (sizeof(R) == 4) {
    // FP32: the real and imaginary parts side by side in the paired FP32
    // instructions (one FFMA2 per matrix entry instead of two FFMAs)
    float2 tot = make_float2(0.0f, 0.0f);
    static_for<0, NC>([&](auto I) {
      constexpr int i = decltype(I)::value;
      constexpr float cii = (float)P::cnum(i, i);
      float2 u = __fmul2_rn(make_float2(cii, cii), make_float2(J[i].re, J[i].im));
      static_for<i + 1, NC>([&](auto Jc) {
        constexpr int j = decltype(Jc)::value;
        if constexpr (P::cnum(i, j) != 0) {
          constexpr float c = (float)(2 * P::cnum(i, j));
          u = __ffma2_rn(make_float2(c, c), make_float2(J[j].re, J[j].im), u);
        }
      });
      tot = __ffma2_rn(make_float2(J[i].re, J[i].im), u, tot);
    });
    return (tot.x + tot.y) / R(P::CDEN);
  }
  R sum = R(0);
  static_for<0, NC>([&](auto I) {
    constexpr int i = decltype(I)::value;
    R ur = R(P::cnum(i, i)) * J[i].re, ui = R(P::cnum(i, i)) * J[i].im;
    static_for<i + 1, NC>([&](auto Jc) {
      constexpr int j = decltype(Jc)::value;
      if constexpr (P::cnum(i, j) != 0) {
        ur = fmac(R(2 * P::cnum(i, j)), J[j].re, ur);
        ui = fmac(R(2 * P::cnum(i, j)), J[j].im, ui);
      }
    });
    sum = fmac(J[i].re, ur, fmac(J[i].im, ui, sum));
  });
  return sum / R(P::CDEN);
}

// Four-point Hadamard transform of every orbit of chains, in place
template <class P, class R>
__device__ __forceinline__ void colour_hadamard(cx<R>* J) {
  static_for<0, 6>([&](auto O) {
    constexpr int o = decltype(O)::value;
    cx<R>&a = J[P::colour_orbit(o, 0)], &b = J[P::colour_orbit(o, 1)], &c = J[P::colour_orbit(o, 2)],
    &d = J[P::colour_orbit(o, 3)];
    const cx<R> ab = a + b, cd = c + d, am = a - b, cm = c - d;
    a = ab + cd;
    b = ab - cd;
    c = am + cm;
    d = am - cm;
  });
}

// |M_h|^2 on CUDA cores: the symmetric form of the whole matrix, or for 24
// flows (where J is left transformed) of its four blocks: 129 paired FP32
// instructions instead of 324 (gg -> t t~ g g, 2^20 events 11.7 -> 10.9 ms)
template <class P, class R>
__device__ __forceinline__ R colour_sum(cx<R>* J) {
  if constexpr (!P::COLOUR_BLOCKS) {
    return colour_sum_sym<P, R>(J);
  } else {
    colour_hadamard<P, R>(J);
    cx<R> tot(R(0), R(0));  // re: sum of the products' real parts; im: of the imaginary parts
    static_for<0, 24>([&](auto I) {
      constexpr int x = decltype(I)::value / 6, i = decltype(I)::value % 6;
      constexpr R mii = (R)P::colour_block(x, i, i);
      const cx<R> y = J[P::colour_orbit(i, x)];
      cx<R> u(mii * y.re, mii * y.im);
      static_for<i + 1, 6>([&](auto Jc) {
        constexpr int j = decltype(Jc)::value;
        if constexpr (P::colour_block(x, i, j) != 0) {
          constexpr R m = (R)(2 * P::colour_block(x, i, j));
          u = pair_fma(cx<R>(m, m), J[P::colour_orbit(j, x)], u);
        }
      });
      tot = pair_fma(y, u, tot);
    });
    return (tot.re + tot.im) / R(4 * P::CDEN);
  }
}

// Propagator factor of one line from its FP64 momentum: the invariant
// k^2 - m^2 is formed in FP64 (it cancels near the pole and for collinear
// pairs); the reciprocal 1/(k^2 - m^2 + i m w) times i (fermion) or -i (vector)
// is taken in the working precision.
template <class R>
__device__ __forceinline__ cx<R> propagator_hs(const double* k, int kind, const PhysParams& pp) {
  const double k2 = k[0] * k[0] - k[1] * k[1] - k[2] * k[2] - k[3] * k[3];
  double dr = k2, di = 0.0;
  if (kind == 1) { dr = k2 - pp.mt * pp.mt; di = pp.mt * pp.wt; }
  else if (kind == 3) { dr = k2 - pp.mz * pp.mz; di = pp.mz * pp.wz; }
  const R r = R(dr), i = R(di);
  const R inv = R(1) / (r * r + i * i);
  const R ar = r * inv, ai = -i * inv;
  return kind == 1 ? cx<R>(-ai, ar) : cx<R>(ai, -ar);
}

// Propagator factor from a double-float momentum: k^2 - m^2 in double-float, then
// the reciprocal in FP32.
// m2 = m^2 as double-float, mw = m w.
template <class V>
__device__ __forceinline__ cx<V> propagator_dfl(const DflSum<V>* k, int kind, dfl m2, float mw) {
  DflSum<V> d = dfl_invariant(k);
  V di(0.0f);
  if (kind == 1 || kind == 3) {
    d.add(V(-m2.hi), V(-m2.lo));
    di = V(mw);
  }
  const V r = d.value();
  const V inv = V(1.0f) / fmac(r, r, di * di);
  const V ar = r * inv, ai = -di * inv;
  return kind == 1 ? cx<V>(-ai, ar) : cx<V>(ai, -ar);
}

// External wavefunctions of the mixed mode, both helicities of a leg from its
// double-float momentum (the formulas of ixxxxx, oxxxxx and vxxxxx): rounded
// once, to FP32.  Near-collinear and soft events amplify the errors of the
// spinors and polarisation vectors; in plain FP32 they were the mixed mode's
// largest error there (2-norm of the error of g g -> t t~ g g over events inside
// generator cuts 6.6e-7, rounded once 4.5e-7).  w[0]: helicity -1, w[1]: +1.
__device__ __forceinline__ void ext_vector_dfl(const dfl* k, int nsv, W4<float>* w) {
  const dfl kt2 = dfl_add(dfl_mul(k[1], k[1]), dfl_mul(k[2], k[2]));
  const dfl kk2 = dfl_add(kt2, dfl_mul(k[3], k[3]));
  const dfl r2 = {0.707106769f, 1.21016175e-8f};  // 1 / sqrt 2
  float x1, x2, x3, y1, y2;  // (ct cp, ct sp, st), (sp, cp) over sqrt 2
  if (kt2.hi > 0.0f) {
    const dfl u = dfl_mul(dfl_rsqrt(kt2), r2), v = dfl_rsqrt(kk2);
    const dfl cp = dfl_mul(k[1], u), sp = dfl_mul(k[2], u), ct = dfl_mul(k[3], v);
    x1 = dfl_value(dfl_mul(ct, cp));
    x2 = dfl_value(dfl_mul(ct, sp));
    x3 = dfl_value(dfl_mul(dfl_mul(kt2, u), v));
    y1 = dfl_value(sp);
    y2 = dfl_value(cp);
  } else {
    x1 = k[3].hi >= 0.0f ? r2.hi : -r2.hi;
    x2 = x3 = y1 = 0.0f;
    y2 = r2.hi;
  }
  const float b = nsv > 0 ? -1.0f : 1.0f;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float a = h == 0 ? 1.0f : -1.0f;
    w[h].w[0] = cx<float>(0.0f, 0.0f);
    w[h].w[1] = cx<float>(a * x1, -b * y1);
    w[h].w[2] = cx<float>(a * x2, b * y2);
    w[h].w[3] = cx<float>(-a * x3, 0.0f);
  }
}
__device__ __forceinline__ void ext_fermion_dfl(const dfl* p, float m, int nsf, bool row, W4<float>* w) {
  const dfl pt2 = dfl_add(dfl_mul(p[1], p[1]), dfl_mul(p[2], p[2]));
  const dfl pp2 = dfl_add(pt2, dfl_mul(p[3], p[3]));
  dfl pp = {0.0f, 0.0f};
  if (pp2.hi > 0.0f) pp = dfl_mul(pp2, dfl_rsqrt(pp2));
  const dfl ppz = p[3].hi >= 0.0f ? dfl_add(pp, p[3])
                                  : dfl_mul(pt2, dfl_rcp(dfl_add(pp, dfl{-p[3].hi, -p[3].lo})));
  // chi_+ = (a, b), chi_- = (-b^*, a), b = (bx, by)
  dfl a = {0.0f, 0.0f}, bx = {1.0f, 0.0f}, by = {0.0f, 0.0f};  // exactly along -z
  if (ppz.hi > 0.0f) {
    const dfl n = dfl_mul(pp, ppz);
    const dfl nrm = dfl_rsqrt(dfl{2.0f * n.hi, 2.0f * n.lo});
    a = dfl_mul(ppz, nrm);
    bx = dfl_mul(p[1], nrm);
    by = dfl_mul(p[2], nrm);
  }
  const dfl e = dfl_add(p[0], pp), r = dfl_rsqrt(e);
  const dfl wp = dfl_mul(e, r), wm = dfl_mul(r, dfl{m, 0.0f});
  float q[2][3];  // omega_+ and omega_- times (a, bx, by)
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const dfl o = i == 0 ? wp : wm;
    q[i][0] = dfl_value(dfl_mul(o, a));
    q[i][1] = dfl_value(dfl_mul(o, bx));
    q[i][2] = dfl_value(dfl_mul(o, by));
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    // u: chi_hel, omegas (-hel, hel); v: chi_-hel, omegas (-hel omega_hel, hel omega_-hel)
    const bool plus = h == 1, chip = nsf > 0 ? plus : !plus;
    const int lo = nsf > 0 ? (plus ? 1 : 0) : (plus ? 0 : 1);
    const float slo = nsf > 0 ? 1.0f : (plus ? -1.0f : 1.0f), shi = nsf > 0 ? 1.0f : -slo;
    cx<float> c[4];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float* z = lo == i ? q[0] : q[1];
      const float s = i == 0 ? slo : shi;
      c[2 * i] = chip ? cx<float>(s * z[0], 0.0f) : cx<float>(-s * z[1], s * z[2]);
      c[2 * i + 1] = chip ? cx<float>(s * z[1], s * z[2]) : cx<float>(s * z[0], 0.0f);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) w[h].w[i] = row ? conj(c[(i + 2) & 3]) : c[i];
  }
}

// The same in FP64: the arithmetic of ixxxxx, oxxxxx and vxxxxx, its square roots
// and quotients (most of the work in FP64) formed once for both helicities.
__device__ __forceinline__ void ext_vector_fp64(const double* k, int nsv, W4<double>* w) {
  const double kt = sqrt(k[1] * k[1] + k[2] * k[2]);
  const double kk = sqrt(kt * kt + k[3] * k[3]);
  double ct, st, cp, sp;
  if (kt == 0.0) { ct = k[3] >= 0.0 ? 1.0 : -1.0; st = 0.0; cp = 1.0; sp = 0.0; }
  else { ct = k[3] / kk; st = kt / kk; cp = k[1] / kt; sp = k[2] / kt; }
  const double r2 = 0.70710678118654752440, b = nsv > 0 ? -r2 : r2;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const double a = h == 0 ? r2 : -r2;
    w[h].w[0] = cx<double>(0.0, 0.0);
    w[h].w[1] = cx<double>(a * ct * cp, b * -sp);
    w[h].w[2] = cx<double>(a * ct * sp, b * cp);
    w[h].w[3] = cx<double>(-a * st, 0.0);
  }
}
__device__ __forceinline__ void ext_fermion_fp64(const double* p, double m, int nsf, bool row, W4<double>* w) {
  cx<double> p0, p1;
  helicity_chi(p, 1, p0, p1);
  // chi_- = (-conj(c1), c0) of chi_+ = (c0, c1), c0 real
  const cx<double> m0(-p1.re, p1.im), m1(p0.re, 0.0);
  double wp, wm;
  omegas(p, m, wp, wm);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const bool plus = h == 1, chip = nsf > 0 ? plus : !plus;
    const cx<double> c0 = chip ? p0 : m0, c1 = chip ? p1 : m1;
    const double lo = nsf > 0 ? (plus ? wm : wp) : (plus ? -wp : wm);
    const double hi = nsf > 0 ? (plus ? wp : wm) : (plus ? wm : -wp);
    const cx<double> c[4] = {lo * c0, lo * c1, hi * c0, hi * c1};
#pragma unroll
    for (int i = 0; i < 4; ++i) w[h].w[i] = row ? conj(c[(i + 2) & 3]) : c[i];
  }
}

// Phase 1 of the forward kernels, in three parts:
//   hs_setup_words   per-CTA constants: {momentum entry, line kind} per
//                    propagator, a descriptor per momentum-table entry, and in
//                    the mixed mode {m^2 hi, m^2 lo, m w, 0} of the top and Z;
//   hs_load_momenta  the CTA's momenta into shared memory: FP64, or in the
//                    mixed mode each component split into a double-float pair;
//   hs_tables        (after a barrier) one thread per (unit, momentum-table
//                    entry) sums the entry's signed external momenta — in FP64
//                    (FP64 mode) or double-float (mixed mode), every leg in leg
//                    order with coefficient +1, -1 or 0 (adding an exact zero
//                    changes neither an FP64 sum nor a double-float pair), rounds
//                    it to R for the currents and forms the propagator factor
//                    of every line with that momentum from the unrounded sum;
//                    one thread per (event, external leg) builds the external
//                    wavefunctions of both helicities (level 0 of the program).

// Descriptor of momentum-table entry j: {legs added, legs subtracted, first
// propagator on that momentum, second} (-1: none).
template <class P>
__device__ __forceinline__ int4 hs_mom_desc(int j) {
  int4 v = make_int4(0, 0, -1, -1);
#pragma unroll
  for (int jj = 0; jj < P::NMOM; ++jj) {
    if (j != jj) continue;
    const int legs = P::mom(jj, 1), neg = P::mom(jj, 0) == 1 ? (P::mom(jj, 2) & legs) : 0;
    v = make_int4(legs & ~neg, neg, P::mom_prop(jj, 0), P::mom_prop(jj, 1));
  }
  return v;
}

template <class P, class R, class L>
__device__ __forceinline__ void hs_setup_words(unsigned char* smem, const PhysParams& pp) {
  static_assert(L::NT >= P::NPROP && L::NT >= P::NMOM, "one thread per propagator and per momentum entry");
  const int tid = threadIdx.x;
  if (tid < P::NPROP) {
    int2 v = make_int2(0, 0);
#pragma unroll
    for (int j = 0; j < P::NPROP; ++j)
      if (tid == j) v = make_int2(P::prop(j, 0), P::prop(j, 1));
    reinterpret_cast<int2*>(smem + L::o_proptab)[tid] = v;
  }
  if (tid < P::NMOM) reinterpret_cast<int4*>(smem + L::o_md)[tid] = hs_mom_desc<P>(tid);
  if constexpr (sizeof(R) == 4) {
    if (tid < 2) {
      const double m = tid == 0 ? pp.mt : pp.mz, w = tid == 0 ? pp.wt : pp.wz;
      const dfl m2 = dfl_split(m * m);
      reinterpret_cast<float4*>(smem + L::o_mconst)[tid] = make_float4(m2.hi, m2.lo, (float)(m * w), 0.0f);
    }
  }
}

// p[unit][leg][mu]: double, or in the mixed mode {hi, lo} of the unit's events
// (EW high parts, then EW low parts); a last unit that is not full repeats its event
template <class P, class R, class L>
__device__ __forceinline__ void hs_put_momentum(unsigned char* smem, int e, int c, int nev, double x) {
  if constexpr (sizeof(R) == 4) {
    constexpr int EW = L::EW;
    const dfl q = dfl_split(x);
    float* d = reinterpret_cast<float*>(smem + L::o_p) + ((e / EW) * P::NPAR * 4 + c) * 2 * EW + e % EW;
    d[0] = q.hi;
    d[EW] = q.lo;
    if (EW == 2 && e == nev - 1 && e % EW == 0) {
      d[1] = q.hi;
      d[EW + 1] = q.lo;
    }
  } else {
    reinterpret_cast<double*>(smem + L::o_p)[e * P::NPAR * 4 + c] = x;
  }
}

template <class P, class R, class L>
__device__ __forceinline__ void hs_load_momenta(unsigned char* smem, const double* __restrict__ mom, int64_t nevt,
                                                int64_t e0, int nev) {
  for (int t = threadIdx.x; t < nev * P::NPAR * 4; t += L::NT) {
    const int e = t % nev, c = t / nev;
    hs_put_momentum<P, R, L>(smem, e, c, nev, mom[(int64_t)c * nevt + e0 + e]);
  }
}

// A later group's momenta, copied asynchronously (cp.async, 8 bytes per
// component) into the staging buffer in the layout of p; the copies of each
// thread complete at its cp_async_wait_all, and hs_convert_momenta (after a
// barrier) turns them into p.
template <class P, class L>
__device__ __forceinline__ void hs_prefetch_momenta(unsigned char* smem, const double* __restrict__ mom, int64_t nevt,
                                                    int64_t e0, int nev) {
  const uint32_t st = tc::smem_addr(smem + L::o_ps);
  for (int t = threadIdx.x; t < nev * P::NPAR * 4; t += L::NT) {
    const int e = t % nev, c = t / nev;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(st + 8u * (uint32_t)(e * P::NPAR * 4 + c)),
                 "l"(mom + (int64_t)c * nevt + e0 + e)
                 : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <class P, class R, class L>
__device__ __forceinline__ void hs_convert_momenta(unsigned char* smem, int nev) {
  const double* st = reinterpret_cast<const double*>(smem + L::o_ps);
  for (int t = threadIdx.x; t < nev * P::NPAR * 4; t += L::NT) {
    hs_put_momentum<P, R, L>(smem, t / (P::NPAR * 4), t % (P::NPAR * 4), nev, st[t]);
  }
}

// CUR_EV: 16-byte words from one unit's current variants to the next's; KEV:
// momentum-table entries (V) from one unit's table to the next's.
template <class P, class R, class L, class V = R, int CUR_EV = P::HS_NSLOT * Slots<V, 1>::NPL, int KEV = 4 * P::NMOM>
__device__ __forceinline__ void hs_tables(unsigned char* smem, const PhysParams& pp, int nev, uint4* curs,
                                          const Couplings<R>& cp) {
  constexpr int NM = P::NMOM, NPAR = P::NPAR, EW = LaneOf<V>::EW;
  constexpr int NEXT = P::hs_level(1);  // external variants
  constexpr bool DF = sizeof(R) == 4;
  const int4* md = reinterpret_cast<const int4*>(smem + L::o_md);
  const int2* prop_tab = reinterpret_cast<const int2*>(smem + L::o_proptab);
  const int nu = (nev + EW - 1) / EW, nep = nu * EW;
  // one thread per (event, leg), both helicities (consecutive items), and one per
  // (unit, momentum entry); the wavefunctions, the longer work, first
  static_assert(NEXT == 2 * NPAR, "level 0: two helicities per leg");
  constexpr int NE = NPAR;
  // the entries begin with a warp of their own (the two kinds of work do not
  // share a warp) where that takes no further round
  const int ne32 = (nep * NE + 31) / 32 * 32, t0 = ne32 + nu * NM <= L::NT ? ne32 : nep * NE;
  for (int t = threadIdx.x; t < t0 + nu * NM; t += L::NT) {
    if (t >= t0) {
      const int t2 = t - t0, u = t2 / NM, j = t2 - u * NM;
      const int4 d = md[j];
      V* const Kj = reinterpret_cast<V*>(smem + L::o_K) + u * KEV + 4 * j;
      cx<V>* const pru = reinterpret_cast<cx<V>*>(smem + L::o_pr) + u * P::NPROP;
      if constexpr (DF) {
        struct alignas(sizeof(V) * 2) HiLo { V hi, lo; };
        const HiLo* q = reinterpret_cast<const HiLo*>(smem + L::o_p) + u * NPAR * 4;
        DflSum<V> k[4];
        alignas(16) V kv[4];
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
          k[mu].first(V(0.0f), V(0.0f));
#pragma unroll
          for (int l = 0; l < NPAR; ++l) {
            const HiLo v = q[l * 4 + mu];
            const V c((d.x >> l & 1) ? 1.0f : ((d.y >> l & 1) ? -1.0f : 0.0f));
            k[mu].add(c * v.hi, c * v.lo);
          }
          kv[mu] = k[mu].value();
        }
#pragma unroll
        for (int i = 0; i < (int)(4 * sizeof(V) / 16); ++i)
          reinterpret_cast<uint4*>(Kj)[i] = reinterpret_cast<const uint4*>(kv)[i];
        const float4* mc = reinterpret_cast<const float4*>(smem + L::o_mconst);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int pj = i == 0 ? d.z : d.w;
          if (pj < 0) continue;
          const int kind = prop_tab[pj].y;
          const float4 c = mc[kind == 3 ? 1 : 0];  // {m^2 hi, m^2 lo, m w, 0} of the top / the Z
          pru[pj] = propagator_dfl<V>(k, kind, dfl{c.x, c.y}, c.z);
        }
      } else {
        const double* q = reinterpret_cast<const double*>(smem + L::o_p) + u * NPAR * 4;
        double k[4];
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
          double s = 0.0;
#pragma unroll
          for (int l = 0; l < NPAR; ++l) {
            const double c = (d.x >> l & 1) ? 1.0 : ((d.y >> l & 1) ? -1.0 : 0.0);
            s += c * q[l * 4 + mu];
          }
          k[mu] = s;
          Kj[mu] = R(s);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int pj = i == 0 ? d.z : d.w;
          if (pj < 0) continue;
          pru[pj] = propagator_hs<R>(k, prop_tab[pj].y, pp);
        }
      }
    } else if (t < nep * NE) {
      const int e = t / NE, j = t - e * NE, u = e / EW, lane = e - u * EW;
      const HsSlots<P, V, P::HS_NSLOT> cur{curs + u * CUR_EV};
      const HsItem it = P::hs_items()[2 * j];
      W4<R> o[2];
      if constexpr (DF) {
        dfl k[4];
#pragma unroll
        for (int mu = 0; mu < 4; ++mu) {
          const float* v =
              reinterpret_cast<const float*>(smem + L::o_p) + ((u * NPAR + it.a) * 4 + mu) * 2 * EW + lane;
          k[mu] = dfl{v[0], v[EW]};
        }
        if (it.type == 2) ext_vector_dfl(k, it.c, o);
        else ext_fermion_dfl(k, it.flag ? cp.mt : 0.0f, it.c, it.type == 1, o);
      } else {
        const double* k = reinterpret_cast<const double*>(smem + L::o_p) + (e * NPAR + it.a) * 4;
        if (it.type == 2) ext_vector_fp64(k, it.c, o);
        else ext_fermion_fp64(k, it.flag ? cp.mt : 0.0, it.c, it.type == 1, o);
      }
      cur.set_lane(it.out, lane, o[0]);
      cur.set_lane(P::hs_items()[2 * j + 1].out, lane, o[1]);
    }
  }
  __syncthreads();
}

// a shared-memory word read where it is written here (not kept in a register)
__device__ __forceinline__ int lds_again(const int* p) { return *reinterpret_cast<const volatile int*>(p); }

// Events per group (whole units of ew): the most a CTA takes at once, or fewer
// where one round spreads the batch over the grid's CTAs (a small batch has one
// unit per CTA instead of a few full CTAs).  With more than one round full groups
// are kept: their warps are full.
__device__ __forceinline__ int hs_events_per_group(int64_t n, int most, int ew) {
  const int g = (int)gridDim.x;
  if (n >= (int64_t)g * most) return most;
  return min(most, ((int)n + g * ew - 1) / (g * ew) * ew);
}

// Item of work index t when the lanes take items item-major: consecutive
// lanes take one item for each of the group's units, so that a warp holds
// 32 / units items (of one vertex type wherever the generator's per-event type
// segments are multiples of that) and reads each descriptor once for all
// its units.
template <class L>
__device__ __forceinline__ int hs_item_of(int t, int nu) {
  // t / nu: t nu < 2^32, so the high word of t times ceil(2^32 / nu) is exact
  return nu == L::EVCAP ? t / L::EVCAP : (nu == 1 ? t : (int)__umulhi((unsigned)t, 0xffffffffu / (unsigned)nu + 1u));
}

// Lanes per item of a phase: one per unit.  Where a process has so few items that
// one round holds eight lanes of each, no fewer than eight: a warp then has four
// variants of one current, where a warp of 32 items would go through every vertex
// type one after the other (64 gg -> t t~ events FP64, one per CTA, 22.1 -> 17.6 us;
// with sixteen lanes 20.0 us, twice the warps in the FP64 pipe.  64 e+e- -> mu+mu-
// events FP64 18.5 -> 14.1 us).
template <class P, class L>
__host__ __device__ constexpr bool hs_few_items() {
  int most = P::HS_NITEM - P::hs_level(P::HS_NLEVEL);
  for (int l = 1; l < P::HS_NLEVEL; ++l) {
    const int n = P::hs_level(l + 1) - P::hs_level(l);
    if (n > most) most = n;
  }
  return L::EVCAP >= 8 && 8 * most <= L::NT;
}
template <class P, class L>
__host__ __device__ constexpr int hs_lanes(int nu) {
  return hs_few_items<P, L>() && nu < 8 ? 8 : nu;
}

// Items of the ordered program: a two-leg current ...
template <class P, class R>
__device__ __forceinline__ void ord_item(const HsItem& it, const HsSlots<P, R, P::HS_NSLOT>& cur, const R* K,
                                         const cx<R>* pr, const Couplings<R>& cp) {
  W4<R> o;
  switch (it.type) {
    case 15: o = FFV1_2<R>(cur[it.in[0]], cur[it.in[1]], R(1), K + 4 * it.k0, cp.mt, pr[it.prop]); break;
    case 16: o = FFV1_1<R>(cur[it.in[0]], cur[it.in[1]], R(1), K + 4 * it.k0, cp.mt, pr[it.prop]); break;
    case 17: o = w4_rscale(vector_pair(cur[it.in[0]], cur[it.in[1]]), -pr[it.prop].im); break;
    default: o = w4_rscale(ord_v3(cur[it.in[0]], cur[it.in[1]], K + 4 * it.k0, K + 4 * it.k1), pr[it.prop].im);
  }
  cur.set(it.out, o);
}
// ... and an operand of the contractions
template <class P, class R>
__device__ __forceinline__ void ord_xitem(const HsItem& it, const HsSlots<P, R, P::HS_NSLOT>& cur,
                                          const HsSlots<P, R, P::HS_XCAP>& xb, const R* K, const cx<R>* pr,
                                          const Couplings<R>& cp) {
  if (it.type == 25) {
    xb.set_scalar(it.out, vdot(cur[it.in[0]], cur[it.in[1]]));
    return;
  }
  W4<R> o, o2;
  if (it.type <= 21) {  // two words
    const HsItemExt ext = P::hs_item_ext()[it.in3()];
    if (P::HS_FOUR && it.type == 21) {
      ord_g3(cur[it.in[0]], cur[it.in[1]], cur[it.in[2]], cur[ext.in[0]], cur[ext.in[1]], cur[ext.in[2]], K, ext.k,
             pr[it.prop].im, o, o2);
    } else if (P::HS_FOUR && it.type == 19) {
      const W4<R> c = row_slash(cur[it.in[2]], cur[ext.in[2]]);
      const cx<R> s = mul_i(pr[it.prop]);
      o = scale(row_kslash_m(w4_add(row_slash(cur[it.in[0]], cur[it.in[1]]), c), K + 4 * it.k0, cp.mt), s);
      o2 = scale(row_kslash_m(w4_sub(row_slash(cur[ext.in[0]], cur[ext.in[1]]), c), K + 4 * it.k0, cp.mt), s);
    } else {
      const W4<R> c = slash_col(cur[ext.in[2]], cur[it.in[2]]);
      o = w4_add(slash_col(cur[it.in[1]], cur[it.in[0]]), c);
      o2 = w4_sub(slash_col(cur[ext.in[1]], cur[ext.in[0]]), c);
    }
    xb.set(it.out + HS_WORD, o2);
  } else if (P::HS_FOUR && it.type == 22) {
    const W4<R> g = ord_v3(cur[it.in[2]], cur[it.in3()], K + 4 * it.k0, K + 4 * it.k1);
    o = w4_lower(w4_sub(vector_pair(cur[it.in[0]], cur[it.in[1]]), g));
  } else if (it.type == 23) {
    o = w4_lower(vector_pair(cur[it.in[0]], cur[it.in[1]]));
  } else {
    o = ord_v3(cur[it.in[0]], cur[it.in[1]], K + 4 * it.k0, K + 4 * it.k1);  // times -1, lower index
    o.w[0] = -o.w[0];
  }
  xb.set(it.out, o);
}

// one current variant (external wavefunctions: hs_tables)
template <class P, class R>
__device__ __forceinline__ void hs_item(const HsItem& it, const Slots<R, P::HS_NSLOT>& cur, const R* K,
                                        const cx<R>* pr, const Couplings<R>& cp) {
  W4<R> o;
  switch (it.type) {
    case 3: o = FFV1_2<R>(cur[it.in[0]], cur[it.in[1]], cp.gs, K + 4 * it.k0, cp.mt, pr[it.prop]); break;
    case 4: o = FFV1_1<R>(cur[it.in[0]], cur[it.in[1]], cp.gs, K + 4 * it.k0, cp.mt, pr[it.prop]); break;
    case 5: o = FFV1P0_3<R>(cur[it.in[0]], cur[it.in[1]], it.a ? cp.ee : cp.gs, pr[it.prop]); break;
    case 6: o = FFV2_4_3<R>(cur[it.in[0]], cur[it.in[1]], cp.gz, cp.gzl, cp.gzr, pr[it.prop]); break;
    case 7: o = VVV1P0_1<R>(cur[it.in[0]], cur[it.in[1]], K + 4 * it.k0, K + 4 * it.k1, cp.gs, pr[it.prop]); break;
    default: {  // four-gluon term X_0 (X_1 . W) - X_1 (X_0 . W), in = {X_0, X_1, W}
      const W4<R> x0 = cur[it.in[0]], x1 = cur[it.in[1]], w = cur[it.in[2]];
      o = vvvv_comb(x0, vdot(x1, w), x1, vdot(x0, w), mul_mi(cp.gs2 * pr[it.prop]));
    }
  }
  cur.set(it.out, o);
}

// one amputated-current variant (reads the currents, writes an operand slot)
template <class P, class R>
__device__ __forceinline__ void hs_xitem(const HsItem& it, const Slots<R, P::HS_NSLOT>& cur,
                                         const Slots<R, P::HS_XCAP>& xb, const R* K, const Couplings<R>& cp) {
  W4<R> o;
  switch (it.type) {
    case 9: o = FFV1_2A<R>(cur[it.in[0]], cur[it.in[1]], cp.gs); break;
    case 10: o = FFV1_1A<R>(cur[it.in[0]], cur[it.in[1]], cp.gs); break;
    case 11: o = FFV1P0_3A<R>(cur[it.in[0]], cur[it.in[1]], it.a ? cp.ee : cp.gs); break;
    case 12: o = FFV2_4_3A<R>(cur[it.in[0]], cur[it.in[1]], cp.gz, cp.gzl, cp.gzr); break;
    case 13: o = VVV1P0_1A<R>(cur[it.in[0]], cur[it.in[1]], K + 4 * it.k0, K + 4 * it.k1, cp.gs); break;
    default: {  // four-gluon term, as in hs_item
      const W4<R> x0 = cur[it.in[0]], x1 = cur[it.in[1]], w = cur[it.in[2]];
      o = vvvv_comb_a(x0, vdot(x1, w), x1, vdot(x0, w), cp.gs2);
    }
  }
  xb.set(it.out, o);
}

// Inverse-CDF sampling by one warp: the first k < n, in order, whose running
// sum of the weights get(k) exceeds u * (their total), the last one if
// rounding leaves none, -1 if the total is not positive (FP64; n <= 32 RND,
// lanes take consecutive k, running sums by warp scans 32 weights at a time,
// the total is the last running sum).
template <int RND, class F>
__device__ __forceinline__ int warp_inverse_cdf(int n, double u, int lane, F get) {
  double run[RND];
  double carry = 0.0;
#pragma unroll
  for (int r = 0; r < RND; ++r) {
    run[r] = 0.0;
    if (32 * r < n) {
      double x = 32 * r + lane < n ? get(32 * r + lane) : 0.0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      run[r] = carry + x;
      carry = __shfl_sync(0xffffffffu, run[r], 31);
    }
  }
  if (!(carry > 0.0)) return -1;
  const double target = u * carry;
#pragma unroll
  for (int r = 0; r < RND; ++r) {
    const unsigned hit = __ballot_sync(0xffffffffu, 32 * r + lane < n && run[r] > target);
    if (hit) return 32 * r + __ffs(hit) - 1;
  }
  return n - 1;
}

// Per event: a good helicity with probability |M_h|^2 / sum (weights sm2 of
// the event, helicity order) and a colour flow s with probability
// w_s / sum, w_s = sum over the good helicities of |J_s|^2; one warp per event.
// The |J_s|^2 of every (event, helicity) are staged in the dead union region, one
// row each with an odd row stride (lane s of the event's warp sums row entries s over
// the event's helicities, in helicity order, in the working precision; the
// running sums that decide are FP64).
template <class P, class R>
struct HsChoice {
  static constexpr int NCP = P::NCOLOR | 1;
};

template <class P, class R, class L>
__device__ __forceinline__ void hs_choices(const unsigned char* smem, const SigArgs& a, int64_t e0, int nev, int ng,
                                           const int* good, const R* sm2) {
  constexpr int NT = L::NT, NC = P::NCOLOR, NCP = HsChoice<P, R>::NCP;
  static_assert(NC <= 32, "one lane per colour flow");
  static_assert(sizeof(R) * NCP * NT * L::EW <= L::u_bytes, "colour weights overflow their scratch");
  const int tid = threadIdx.x, lane = tid & 31;
  const R* wj = reinterpret_cast<const R*>(smem + L::o_U);
  for (int e = tid >> 5; e < nev; e += NT / 32) {
    if (a.hel_out) {
      const int k = warp_inverse_cdf<(P::NHEL + 31) / 32>(ng, a.hel_rnd[e0 + e], lane,
                                                          [&](int i) { return (double)sm2[e * ng + i]; });
      if (lane == 0) a.hel_out[e0 + e] = k < 0 ? -1 : good[k];
    }
    if (a.col_out) {
      R x = R(0);
      if (lane < NC)
        for (int k = 0; k < ng; ++k) x += wj[(e * ng + k) * NCP + lane];
      const double w = (double)x;
      const int c = warp_inverse_cdf<1>(NC, a.col_rnd[e0 + e], lane, [&](int) { return w; });
      if (lane == 0) a.col_out[e0 + e] = c;
    }
  }
}

// Record of one unit's current variants and momentum tables in global memory
// (the kernel-split variant: the first kernel writes them, the second reads
// them back into shared memory; R the lane type): HS_NSLOT slots of 16-byte planes, then the
// momentum table K[NMOM][4] in the working precision and, where operands of the
// contractions have propagators (ordered program), the propagator factors.
template <class P, class R>
struct HsRecord {
  static constexpr int CUR = P::HS_NSLOT * Slots<R, 1>::NPL;
  static_assert((P::NMOM * 4 * sizeof(R)) % 16 == 0, "momentum table in 16-byte words");
  static constexpr int KW = (int)(P::NMOM * 4 * sizeof(R) / 16);
  static constexpr int PW = P::HS_ORDERED ? (int)(align_up(P::NPROP * sizeof(cx<R>), 16) / 16) : 0;
  static constexpr int WORDS = CUR + KW + PW;
};

// Where a group's momenta come from: the momentum buffer (mg_sigmakin), the
// kernel-split records (current variants and momentum tables instead), or
// RAMBO inside the kernel (mg_sigmakin_rambo, mg_sigmakin_seeded).
constexpr int kSrcMomenta = 0, kSrcRecords = 1, kSrcRambo = 2;

// One event's RAMBO inside a SIGMAKIN kernel: the uniforms as the RAMBO kernel
// reads or draws them, the same forward code (rambo_forward), the momenta of
// all legs into out[leg][mu] (shared memory, FP64; the beams as the RAMBO
// kernel writes them) and the weight into wgt.  Not inlined, so that RAMBO's
// many FP64 temporaries do not raise the register count of the calling
// kernel (the call runs on a few lanes, once per event).
template <int NF>
__device__ __noinline__ void rambo_event_fused(const double* __restrict__ rnd, int64_t nevt, int64_t i, uint64_t key,
                                               int64_t first_event, double ecm, const RamboSetup& st, double* out,
                                               double* __restrict__ wgt) {
  double r[4 * NF];
  if (rnd) {
#pragma unroll
    for (int k = 0; k < 4 * NF; ++k) r[k] = rnd[(int64_t)k * nevt + i];
  } else {
#pragma unroll
    for (int k = 0; k < 4 * NF; ++k) r[k] = sm64_uniform(key, first_event + i, k);
  }
  RamboState<NF> z;
  rambo_forward<NF>(r, ecm, st, z);
  const double h = 0.5 * ecm;
  out[0] = h; out[1] = 0.0; out[2] = 0.0; out[3] = h;
  out[4] = h; out[5] = 0.0; out[6] = 0.0; out[7] = -h;
#pragma unroll
  for (int f = 0; f < NF; ++f)
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) out[(2 + f) * 4 + mu] = z.k[f][mu];
  wgt[i] = z.w;
}

// averaging factors, and the coupling where the currents go without it
template <class P>
__device__ __forceinline__ double hs_norm(const PhysParams& pp) {
  double f = P::NORM;
#pragma unroll
  for (int k = 0; k < P::HS_GS_POWER / 2; ++k) f *= pp.gs2;
  return f;
}

// The helicity-shared program for the events [first, last) of the batch.
// SRC == kSrcRecords: phases 1-2 (momenta, tables, current variants) are
// replaced by a copy of the records from `rec` (one record per unit, the unit of
// event `first` at rec[0]).
template <class P, class R, int CS, int SRC>
__device__ __forceinline__ void hs_sigmakin_body(const SigArgs& a, const Couplings<R>& cp, int64_t first, int64_t last,
                                                 const uint4* __restrict__ rec, const RamboArgs* ra = nullptr) {
  using L = HsLayout<P, R, CS, SRC == kSrcRambo>;
  using V = typename L::V;
  constexpr bool FROM_RECORDS = SRC == kSrcRecords;
  static_assert(!(FROM_RECORDS && L::TC), "the kernel-split variant sums colours on CUDA cores");
  constexpr int NT = L::NT, NC = P::NCOLOR, EW = L::EW;
  extern __shared__ __align__(1024) unsigned char smem[];
  int* good = reinterpret_cast<int*>(smem + L::o_good);
  int* misc = reinterpret_cast<int*>(smem + L::o_misc);
  R* sm2 = reinterpret_cast<R*>(smem + L::o_m2);
  uint8_t* vtab = reinterpret_cast<uint8_t*>(smem + L::o_vt);
  // per unit: HS_NSLOT current slots, HS_XCAP further operands (16-byte planes)
  uint4* curs = reinterpret_cast<uint4*>(smem + L::o_cur);
  uint4* xbufs = reinterpret_cast<uint4*>(smem + L::o_x);
  constexpr int CUR_EV = L::CUR_EV, X_EV = L::X_EV;
  const int tid = threadIdx.x, lane = tid & 31;
  hs_setup_words<P, R, L>(smem, a.pp);
  // vt[row][ihel]: variant index of the row's leg set for helicity ihel (generated table)
  static_assert((P::HS_NVT * P::NHEL) % 16 == 0, "variant table copied in 16-byte words");
  for (int i = tid; i < P::HS_NVT * P::NHEL / 16; i += NT)
    reinterpret_cast<uint4*>(vtab)[i] = reinterpret_cast<const uint4*>(P::hs_variants())[i];
  // good helicities: every warp ballots the mask itself (32 helicities per
  // word), so the events and their momenta are known before any barrier;
  // good[] in helicity order (read only after later barriers)
  static_assert(P::NHEL <= 64 && NT >= P::NHEL, "helicity ballot layout");
  const unsigned w0 = __ballot_sync(0xffffffffu, lane < P::NHEL && a.mask[lane] != 0);
  const unsigned w1 = P::NHEL > 32 ? __ballot_sync(0xffffffffu, lane + 32 < P::NHEL && a.mask[lane + 32] != 0) : 0u;
  if (tid < P::NHEL) {
    const unsigned w = tid < 32 ? w0 : w1, bit = 1u << (tid & 31);
    if (w & bit) good[__popc(w & (bit - 1u)) + (tid >= 32 ? __popc(w0) : 0)] = tid;
  }
  const int ng = __popc(w0) + __popc(w1);
  const int ev = hs_events_per_group(last - first, EW * (ng > 0 ? min(L::EVCAP, NT / ng) : L::H::EVMIN), EW);
  // groups of ev events, g = blockIdx.x, blockIdx.x + gridDim.x, ...: one
  // group per CTA for a grid of all groups, several for a persistent grid
  const int ngrp = (int)((last - first + ev - 1) / ev);
  if ((int)blockIdx.x >= ngrp) return;
  // kept in shared memory and read where they are needed: registers that would
  // stay live through the contractions otherwise
  if (tid == 0) {
    misc[2] = ngrp;
    misc[6] = ng;
    misc[7] = ev;
    *reinterpret_cast<double*>(misc + 8) = hs_norm<P>(a.pp);
  }
  if (ng == 0) {
    for (int g = blockIdx.x; g < ngrp; g += gridDim.x) {
      const int64_t e0 = first + (int64_t)g * ev;
      if (tid < (int)min((int64_t)ev, last - e0)) {
        a.me[e0 + tid] = 0.0;
        if (a.hel_out) a.hel_out[e0 + tid] = -1;
        if (a.col_out) a.col_out[e0 + tid] = -1;
        if constexpr (SRC == kSrcRambo)  // the weight all the same
          rambo_event_fused<P::NPAR - 2>(ra->rnd, a.nevt, e0 + tid, ra->key, ra->first_event, ra->ecm, ra->st,
                                         reinterpret_cast<double*>(smem + L::o_ps) + tid * P::NPAR * 4, ra->wgt);
      }
    }
    return;
  }
  uint32_t tmem = 0, mbar = 0;
  if constexpr (L::TC) {
    if (tid < 32) tc::tmem_alloc(tc::smem_addr(misc + 1), L::TMEM_COLS);
    mbar = tc::smem_addr(misc + 4);
    if (tid == 0) tc::mbar_init(mbar, 1);
    tc::fence_async_shared();
    tc::fence_before_sync();
  }
  const V* Kall = reinterpret_cast<const V*>(smem + L::o_K);
  const cx<V>* prall = reinterpret_cast<const cx<V>*>(smem + L::o_pr);
  const Couplings<V> cv = lane_couplings<V>(cp);
  const HsItem* items = P::hs_items();
  if constexpr (SRC == kSrcMomenta) {
    // the first group's momenta; later groups' arrive by prefetch
    const int64_t e0 = first + (int64_t)blockIdx.x * ev;
    hs_load_momenta<P, R, L>(smem, a.mom, a.nevt, e0, (int)min((int64_t)ev, last - e0));
  } else if constexpr (SRC == kSrcRambo) {
    // the first group's RAMBO, one lane per event, into the staging buffer
    const int64_t e0 = first + (int64_t)blockIdx.x * ev;
    const int nev0 = (int)min((int64_t)ev, last - e0);
    if (tid < nev0)
      rambo_event_fused<P::NPAR - 2>(ra->rnd, a.nevt, e0 + tid, ra->key, ra->first_event, ra->ecm, ra->st,
                                     reinterpret_cast<double*>(smem + L::o_ps) + tid * P::NPAR * 4, ra->wgt);
    __syncthreads();
    hs_convert_momenta<P, R, L>(smem, nev0);
  }
  __syncthreads();
  if constexpr (L::TC) {
    tc::fence_after_sync();
    tmem = static_cast<uint32_t>(misc[1]);
  }
#pragma unroll 1
  for (int g = blockIdx.x; g < lds_again(misc + 2); g += gridDim.x) {
    // e0 and nev are formed again after the contractions (fewer live registers)
    const int ev = lds_again(misc + 7);
    const int nev = (int)min((int64_t)ev, last - (first + (int64_t)g * ev));
    const int nu = (nev + EW - 1) / EW;
    constexpr bool FEW = hs_few_items<P, L>();
    const int nl = hs_lanes<P, L>(nu);  // lanes per item
    if constexpr (FROM_RECORDS) {
      // 1-2. the units' current variants and momentum tables from their records
      using RC = HsRecord<P, V>;
      const uint4* in = rec + (int64_t)g * (ev / EW) * RC::WORDS;
      uint4* ks = reinterpret_cast<uint4*>(smem + L::o_K);
      for (int t = tid; t < nu * RC::WORDS; t += NT) {
        const int u = t / RC::WORDS, w = t - u * RC::WORDS;
        const uint4 v = __ldcs(in + t);  // read once: streaming
        if (w < RC::CUR) curs[u * CUR_EV + w] = v;
        else if (w < RC::CUR + RC::KW) ks[u * (L::KEV * (int)sizeof(V) / 16) + (w - RC::CUR)] = v;
        else {
          const cx<V>* f = reinterpret_cast<const cx<V>*>(&v);
          constexpr int PER = (int)(16 / sizeof(cx<V>));
#pragma unroll
          for (int k = 0; k < PER; ++k) {
            const int j = (w - RC::CUR - RC::KW) * PER + k;
            if (j < P::NPROP) reinterpret_cast<cx<V>*>(smem + L::o_pr)[u * P::NPROP + j] = f[k];
          }
        }
      }
      __syncthreads();
    } else {
      // the next group's momenta: copied during this group's phases 1-2 and
      // converted after the last current level (p is free once the tables are built)
      const int gn = g + gridDim.x;
      const int64_t e0n = first + (int64_t)gn * ev;
      const int nevn = gn < lds_again(misc + 2) ? (int)min((int64_t)ev, last - e0n) : 0;
      if constexpr (SRC == kSrcRambo) {
        // the next group's RAMBO on the last lanes, which the tables phase
        // leaves idle when it has fewer items than threads
        const int u = NT - 1 - tid;
        if (u < nevn)
          rambo_event_fused<P::NPAR - 2>(ra->rnd, a.nevt, e0n + u, ra->key, ra->first_event, ra->ecm, ra->st,
                                         reinterpret_cast<double*>(smem + L::o_ps) + u * P::NPAR * 4, ra->wgt);
      } else {
        if (nevn > 0) hs_prefetch_momenta<P, L>(smem, a.mom, a.nevt, e0n, nevn);
      }
      // 1. per-event tables (the momenta are in p)
      hs_tables<P, R, L, V, CUR_EV, L::KEV>(smem, a.pp, nev, curs, cp);
      // 2. current variants, level by level (level 0, the external wavefunctions,
      //    came with phase 1); consecutive threads take one item for each event (hs_item_of)
#pragma unroll
      for (int l = 1; l < P::HS_NLEVEL; ++l) {
        const int i0 = P::hs_level(l), n = (P::hs_level(l + 1) - i0) * nl;
        for (int t = tid; t < n; t += NT) {
          const int ii = hs_item_of<L>(t, nl), u = t - ii * nl;
          if (FEW && u >= nu) continue;
          const HsItem it = items[i0 + ii];
          const HsSlots<P, V, P::HS_NSLOT> cur{curs + u * CUR_EV};
          if constexpr (P::HS_ORDERED) ord_item<P, V>(it, cur, Kall + u * L::KEV, prall + u * P::NPROP, cv);
          else hs_item<P, V>(it, cur, Kall + u * L::KEV, prall + u * P::NPROP, cv);
        }
        if (l == P::HS_NLEVEL - 1) {
          cp_async_wait_all();
          __syncthreads();
          if (nevn > 0) hs_convert_momenta<P, R, L>(smem, nevn);
        } else {
          __syncthreads();
        }
      }
    }
    // 3. the operands of the contractions (amputated currents), then every
    //    thread contracts for its (unit, helicity), J in registers
    static_assert(P::HS_NXCHUNK == 1, "the operands of every contraction at once");
    {
      const int i0 = P::hs_xitem(0), n = (P::hs_xitem(1) - i0) * nl;
      for (int t = tid; t < n; t += NT) {
        const int ii = hs_item_of<L>(t, nl), ui = t - ii * nl;
        if (FEW && ui >= nu) continue;
        const HsItem it = items[i0 + ii];
        const HsSlots<P, V, P::HS_NSLOT> cur{curs + ui * CUR_EV};
        const HsSlots<P, V, P::HS_XCAP> xs{xbufs + ui * X_EV};
        if constexpr (P::HS_ORDERED) ord_xitem<P, V>(it, cur, xs, Kall + ui * L::KEV, prall + ui * P::NPROP, cv);
        else hs_xitem<P, V>(it, cur, xs, Kall + ui * L::KEV, cv);
      }
    }
    __syncthreads();
    const int ng = lds_again(misc + 6);
    const bool active = tid < nu * ng;
    const int u = active ? tid / ng : 0, kh = active ? tid - u * ng : 0;  // unit, good helicity
    cx<V> J[NC];
#pragma unroll
    for (int s = 0; s < NC; ++s) J[s] = cx<V>(V(0), V(0));
    P::template hs_contract<V>(0, HsSlots<P, V, P::HS_NSLOT>{curs + u * CUR_EV},
                               HsSlots<P, V, P::HS_XCAP>{xbufs + u * X_EV}, vtab + good[kh], J);
    // the flows' |J_s|^2 for the choice of one (batched entry point), into the union
    // once every thread of the CTA is done with it: from the J of the chains,
    // before the colour sum transforms them (back and forth a small flow would
    // carry the rounding of the largest of its orbit)
    [[maybe_unused]] auto stage_flows = [&] {
      __syncthreads();
      R* wj = reinterpret_cast<R*>(smem + L::o_U);  // rows as sm2's
      if (active) {
#pragma unroll
        for (int i = 0; i < EW; ++i)
#pragma unroll
          for (int s = 0; s < NC; ++s) {
            const R re = lane_value(J[s].re, i), im = lane_value(J[s].im, i);
            wj[((u * EW + i) * ng + kh) * HsChoice<P, R>::NCP + s] = re * re + im * im;
          }
      }
    };
    // (compiled in for every source of momenta, though only mg_matrix_elements_batch
    // asks for choices: the branch also keeps the loads of the contractions where
    // they are.  Without it the kernel with RAMBO inside takes 255 registers and
    // spills, 30011 gg -> t t~ g g events 965 us instead of 871)
    if constexpr (!L::TC)
      if (a.col_out) stage_flows();
    // 4. colour sum and helicity sum; |M_h|^2 of (event, good helicity) k at
    //    sm2[event * ng + k]
    V m2;
    if constexpr (L::TC) {
      __syncthreads();  // the A tiles overwrite the current variants
      m2 = colour_sum_tc_regs<P, L>(smem, J, tmem, mbar);
    } else {
      m2 = colour_sum<P, V>(J);
    }
    if (active) {
#pragma unroll
      for (int i = 0; i < EW; ++i) sm2[(u * EW + i) * ng + kh] = lane_value(m2, i);
    }
    if constexpr (L::TC) tc::fence_before_sync();
    __syncthreads();
    const int64_t e0 = first + (int64_t)g * lds_again(misc + 7);
    // fixed-order FP64 helicity sum per event: eight lanes per event each add
    // every eighth helicity in order, then a butterfly over the eight lanes
    // (addition commutes, so every lane ends with the same bits); sm2 is next
    // written at the end of the next group, after several barriers; the last warps
    // take it, the first ones begin with the next group's wavefunctions
    for (int b = 0; b < nev * 8; b += NT) {
      const int t = b + (NT - 1 - tid), eh = t >> 3, q = t & 7;
      if ((t & ~31) >= nev * 8) continue;  // whole warps without an event
      double sum = 0.0;
      if (t < nev * 8) {
#pragma unroll
        for (int i = 0; i < (P::NHEL + 7) / 8; ++i)
          if (q + 8 * i < ng) sum += (double)sm2[eh * ng + q + 8 * i];
      }
      sum += __shfl_xor_sync(0xffffffffu, sum, 1);
      sum += __shfl_xor_sync(0xffffffffu, sum, 2);
      sum += __shfl_xor_sync(0xffffffffu, sum, 4);
      if (t < nev * 8 && q == 0) a.me[e0 + eh] = sum * *reinterpret_cast<const double*>(misc + 8);
    }
    // 5. helicity and colour-flow choices (batched entry point); the closing
    //    barrier keeps the next group's currents out of the union, and its sm2
    //    unwritten, until the choices are made
    if (SRC == kSrcMomenta && (a.hel_out || a.col_out)) {
      if constexpr (L::TC) {  // the tensor cores have read their tiles
        if (a.col_out) {
          stage_flows();
          __syncthreads();
        }
      }
      hs_choices<P, R, L>(smem, a, e0, nev, ng, good, sm2);
      __syncthreads();
    }
  }
  if constexpr (L::TC) {
    if (tid < 32) {
      tc::fence_after_sync();
      tc::tmem_dealloc(tmem, L::TMEM_COLS);
    }
  }
}

template <class P, class R, int CS>
__global__ void __launch_bounds__(HsCfg<P, R, CS>::NT, HsCfg<P, R, CS>::CTAS) sigmakin_hs_kernel(SigArgs a, Couplings<R> cp) {
  hs_sigmakin_body<P, R, CS, kSrcMomenta>(a, cp, 0, a.nevt, nullptr);
}

// RAMBO and SIGMAKIN in one kernel: no momentum buffer in HBM
template <class P, class R, int CS>
__global__ void __launch_bounds__(HsCfg<P, R, CS, true>::NT, HsCfg<P, R, CS, true>::CTAS)
    sigmakin_hs_rambo_kernel(SigArgs a, Couplings<R> cp, RamboArgs ra) {
  hs_sigmakin_body<P, R, CS, kSrcRambo>(a, cp, 0, a.nevt, nullptr, &ra);
}

}  // namespace mg
