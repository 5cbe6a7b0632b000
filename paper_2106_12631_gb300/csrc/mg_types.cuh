// Complex numbers, wavefunction objects and couplings for the matrix-element
// kernels.  R is the working precision: double (plain FP64 path) or float
// (mixed path).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace mg {

template <class R>
struct cx {
  R re, im;
  cx() = default;
  __host__ __device__ constexpr cx(R r, R i) : re(r), im(i) {}
};
template <class R> __device__ __forceinline__ cx<R> operator+(cx<R> a, cx<R> b) { return cx<R>(a.re + b.re, a.im + b.im); }
template <class R> __device__ __forceinline__ cx<R> operator-(cx<R> a, cx<R> b) { return cx<R>(a.re - b.re, a.im - b.im); }
template <class R> __device__ __forceinline__ cx<R> operator-(cx<R> a) { return cx<R>(-a.re, -a.im); }
template <class R> __device__ __forceinline__ cx<R> operator*(cx<R> a, cx<R> b) {
  return cx<R>(a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re);
}
template <class R> __device__ __forceinline__ cx<R> operator*(R s, cx<R> a) { return cx<R>(s * a.re, s * a.im); }
template <class R> __device__ __forceinline__ cx<R> operator*(cx<R> a, R s) { return cx<R>(s * a.re, s * a.im); }
template <class R> __device__ __forceinline__ cx<R>& operator+=(cx<R>& a, cx<R> b) { a.re += b.re; a.im += b.im; return a; }
template <class R> __device__ __forceinline__ cx<R>& operator-=(cx<R>& a, cx<R> b) { a.re -= b.re; a.im -= b.im; return a; }
template <class R> __device__ __forceinline__ cx<R> conj(cx<R> a) { return cx<R>(a.re, -a.im); }
template <class R> __device__ __forceinline__ cx<R> mul_i(cx<R> a) { return cx<R>(-a.im, a.re); }   // i * a
template <class R> __device__ __forceinline__ cx<R> mul_mi(cx<R> a) { return cx<R>(a.im, -a.re); }  // -i * a
// fused multiply-add in the working precision (one rounding)
template <class R> __device__ __forceinline__ R fmac(R a, R b, R c) {
  if constexpr (sizeof(R) == 4) return __fmaf_rn(a, b, c);
  else return __fma_rn(a, b, c);
}
// a b + c and s a + c as chains of fused multiply-adds (four and two
// operations; a product followed by a separate sum takes six and four)
template <class R> __device__ __forceinline__ cx<R> cfma(cx<R> a, cx<R> b, cx<R> c) {
  return cx<R>(fmac(a.re, b.re, fmac(-a.im, b.im, c.re)), fmac(a.re, b.im, fmac(a.im, b.re, c.im)));
}
template <class R> __device__ __forceinline__ cx<R> rfma(R s, cx<R> a, cx<R> c) {
  return cx<R>(fmac(s, a.re, c.re), fmac(s, a.im, c.im));
}

// Two events side by side: the mixed mode's kernels evaluate a pair of events
// per thread, so that every FP32 operation is one paired instruction (FFMA2,
// FADD2, FMUL2: two results per issue slot; operand signs and a scalar repeated
// in both halves cost nothing).  The arithmetic of each event is that of a
// single float.
struct alignas(8) f2 {
  float x, y;
  f2() = default;
  __host__ __device__ constexpr f2(float a, float b) : x(a), y(b) {}
  __host__ __device__ explicit constexpr f2(float a) : x(a), y(a) {}
  __host__ __device__ explicit constexpr f2(double a) : x((float)a), y((float)a) {}
  __host__ __device__ explicit constexpr f2(int a) : x((float)a), y((float)a) {}
};
__device__ __forceinline__ float2 f2_raw(f2 a) { return make_float2(a.x, a.y); }
__device__ __forceinline__ f2 f2_of(float2 a) { return f2(a.x, a.y); }
__device__ __forceinline__ f2 operator-(f2 a) { return f2(-a.x, -a.y); }
__device__ __forceinline__ f2 operator+(f2 a, f2 b) { return f2_of(__fadd2_rn(f2_raw(a), f2_raw(b))); }
__device__ __forceinline__ f2 operator-(f2 a, f2 b) { return f2_of(__fadd2_rn(f2_raw(a), f2_raw(-b))); }
__device__ __forceinline__ f2 operator*(f2 a, f2 b) { return f2_of(__fmul2_rn(f2_raw(a), f2_raw(b))); }
__device__ __forceinline__ f2& operator+=(f2& a, f2 b) { a = a + b; return a; }
__device__ __forceinline__ f2& operator-=(f2& a, f2 b) { a = a - b; return a; }
__device__ __forceinline__ f2 operator/(f2 a, f2 b) { return f2(a.x / b.x, a.y / b.y); }
__device__ __forceinline__ f2 fmac(f2 a, f2 b, f2 c) { return f2_of(__ffma2_rn(f2_raw(a), f2_raw(b), f2_raw(c))); }
// a product and a sum that are rounded by themselves (dfl.cuh); the paired ones always are
__device__ __forceinline__ f2 mul_rn(f2 a, f2 b) { return a * b; }
__device__ __forceinline__ f2 add_rn(f2 a, f2 b) { return a + b; }
__device__ __forceinline__ cx<f2> operator*(cx<f2> a, cx<f2> b) {
  return cx<f2>(fmac(-a.im, b.im, a.re * b.re), fmac(a.im, b.re, a.re * b.im));
}
// scalar type and events of a lane type; value of one event
template <class V>
struct LaneOf {
  using scalar = V;
  static constexpr int EW = 1;
};
template <>
struct LaneOf<f2> {
  using scalar = float;
  static constexpr int EW = 2;
};
template <class V> __host__ __device__ __forceinline__ V lane_value(V v, int) { return v; }
__host__ __device__ __forceinline__ float lane_value(f2 v, int i) { return i == 0 ? v.x : v.y; }

// Four complex components: a Dirac spinor (chiral basis, upper pair
// left-handed; a row spinor for flowing-out fermions, a column spinor for
// flowing-in ones) or a Lorentz vector with upper index.  The paper's
// six-component wavefunction (Sec. 2) also carries the momentum; here the
// momenta are helicity independent and live in a per-event table instead.
template <class R>
struct alignas(16) W4 {
  cx<R> w[4];
};

// An array of N wavefunction slots stored as 16-byte planes: plane k holds
// bytes [16k, 16k + 16) of every slot.  Threads that read consecutive slots
// then touch consecutive 16-byte words of shared memory (no bank conflicts),
// and threads that read the same slot share one access.
template <class R, int N>
struct Slots {
  static constexpr int NPL = (int)(sizeof(W4<R>) / 16);
  uint4* p;
  __device__ __forceinline__ W4<R> operator[](int i) const {
    W4<R> w;
    uint4* d = reinterpret_cast<uint4*>(&w);
#pragma unroll
    for (int k = 0; k < NPL; ++k) d[k] = p[i + k * N];
    return w;
  }
  __device__ __forceinline__ void set(int i, const W4<R>& w) const {
    const uint4* s = reinterpret_cast<const uint4*>(&w);
#pragma unroll
    for (int k = 0; k < NPL; ++k) p[i + k * N] = s[k];
  }
  // one event's values of a slot (lane of V)
  template <class S>
  __device__ __forceinline__ void set_lane(int i, int lane, const W4<S>& w) const {
    constexpr int EW = LaneOf<R>::EW, PER = (int)(16 / sizeof(R));
    const S* v = reinterpret_cast<const S*>(&w);
#pragma unroll
    for (int k = 0; k < 8; ++k) reinterpret_cast<S*>(p + i + (k / PER) * N)[(k % PER) * EW + lane] = v[k];
  }
  // slot i += w, component by component with shared-memory atomics (adjoint
  // accumulation from many threads)
  __device__ __forceinline__ void atomic_add(int i, const W4<R>& w) const {
    constexpr int PER = (int)(16 / sizeof(R));  // values per 16-byte plane word
    const R* s = reinterpret_cast<const R*>(&w);
#pragma unroll
    for (int k = 0; k < NPL; ++k) {
      R* d = reinterpret_cast<R*>(p + i + k * N);
#pragma unroll
      for (int q = 0; q < PER; ++q) atomicAdd(d + q, s[k * PER + q]);
    }
  }
};

// The ordered program's slots: the real parts of a wavefunction's four
// components, then the imaginary parts, so that the components come in
// register pairs for the paired FP32 instructions (dot4p).  After the N slots
// of a region, its scalars.
template <class R, int N>
struct PlanarSlots {
  static constexpr int NPL = (int)(sizeof(W4<R>) / 16), PER = (int)(16 / sizeof(R));
  uint4* p;
  __device__ __forceinline__ W4<R> operator[](int i) const {
    alignas(16) R v[8];
#pragma unroll
    for (int k = 0; k < NPL; ++k) *reinterpret_cast<uint4*>(v + k * PER) = p[i + k * N];
    W4<R> w;
#pragma unroll
    for (int c = 0; c < 4; ++c) w.w[c] = cx<R>(v[c], v[4 + c]);
    return w;
  }
  __device__ __forceinline__ void set(int i, const W4<R>& w) const {
    alignas(16) R v[8];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      v[c] = w.w[c].re;
      v[4 + c] = w.w[c].im;
    }
#pragma unroll
    for (int k = 0; k < NPL; ++k) p[i + k * N] = *reinterpret_cast<const uint4*>(v + k * PER);
  }
  template <class S>
  __device__ __forceinline__ void set_lane(int i, int lane, const W4<S>& w) const {
    constexpr int EW = LaneOf<R>::EW;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const S v = c < 4 ? w.w[c & 3].re : w.w[c & 3].im;
      reinterpret_cast<S*>(p + i + (c / PER) * N)[(c % PER) * EW + lane] = v;
    }
  }
  __device__ __forceinline__ cx<R> scalar(int i) const { return reinterpret_cast<const cx<R>*>(p + N * NPL)[i]; }
  __device__ __forceinline__ void set_scalar(int i, cx<R> x) const { reinterpret_cast<cx<R>*>(p + N * NPL)[i] = x; }
};

// Couplings and masses in the working precision.
template <class R>
struct Couplings {
  R gs;    // strong coupling g_s (quark-gluon i g_s gamma^mu T^a, three-gluon g_s f^abc [..])
  R gs2;   // g_s^2 (four-gluon -i g_s^2 [..])
  R ee;    // e; photon-lepton vertex -i e Q gamma^mu with Q = -1
  R gz;    // e / (sin theta_W cos theta_W)
  R gzl;   // Z left coupling of charged leptons, T3 - Q sin^2 theta_W
  R gzr;   // Z right coupling, -Q sin^2 theta_W
  R mt;    // top mass
};

template <class V, class S>
__device__ __forceinline__ Couplings<V> lane_couplings(const Couplings<S>& c) {
  return {V(c.gs), V(c.gs2), V(c.ee), V(c.gz), V(c.gzl), V(c.gzr), V(c.mt)};
}

// Helicity-shared program tables (generated per process).
// One variant of one off-shell current or amputated current: type (0 ixxxxx,
// 1 oxxxxx, 2 vxxxxx, 3 off-shell flowing-out fermion, 4 off-shell flowing-in
// fermion, 5 vector from a fermion pair, 6 Z from a lepton pair, 7 three-gluon,
// 8 four-gluon term; amputated: 9 row, 10 column, 11 fermion pair, 12 lepton
// pair to Z, 13 three-gluon, 14 four-gluon term); a/b/c: type parameters
// (external: leg, helicity, flow sign; pair: coupling 0 g_s / 1 e); flag:
// external top mass; out/in: variant slots (a four-gluon term's three
// operands X_0, X_1, W); k0/k1: momentum-table entries; prop: propagator
// entry.  One aligned 16-byte word, read by one load.
// Ordered program (types 15 on, see helas.cuh): 15 R(a), 16 C(a), 17 V, 18
// G(ab), 19 R(ab) and R(ba), 20 C(ab) and C(ba), 21 G(ijk) and G(ikj), 22 vector
// vertex B, 23 W, 24 P, 25 scalar product; a fourth operand, or the index of
// the item's extension, in place of a and b (in3); an item with two words
// writes the second one HS_WORD slots after the first.
constexpr int HS_WORD = 8;
struct alignas(16) HsItem {
  uint16_t out;
  uint16_t in[3];
  uint8_t type;
  int8_t a, b, c;
  uint8_t flag, k0, k1, prop;
  __host__ __device__ int in3() const { return (uint8_t)a | (uint8_t)b << 8; }
};
static_assert(sizeof(HsItem) == 16, "item descriptor: one 16-byte word");
// Further operand slots of an item with two words, and for three gluons the
// momentum entries of i, j, k, ij, ik, jk.
struct alignas(16) HsItemExt {
  uint16_t in[3];
  uint8_t k[6];
};
// Physics parameters in FP64 (propagator denominators are formed in FP64 in
// both precision modes); gs2 = g_s^2.
struct PhysParams {
  double mz, wz, mt, wt, gs2;
};

}  // namespace mg
