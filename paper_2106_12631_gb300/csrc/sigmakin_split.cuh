// Kernel-split variant of the helicity-shared program (the outlook of
// Sec. 4: SIGMAKIN split into smaller kernels orchestrated with CUDA Graphs,
// to relieve the one large kernel).  Two kernels per chunk of events:
//   currents:   momenta -> tables -> external wavefunctions -> every current
//               variant (phases 1-2 of the helicity-shared kernel), written
//               as one record per event (HsRecord) to a chunk buffer;
//   amplitudes: the records back into shared memory, then phases 3-5 of the
//               helicity-shared kernel (amputated currents, contractions,
//               colour sum on CUDA cores, helicity sum, choices).
// Chunks small enough that two chunk buffers stay in L2 alternate, so that the
// currents of chunk c + 1 run beside the amplitudes of chunk c; the launches
// of a whole batch are captured once into a CUDA graph (split_graph.cu).
#pragma once
#include <algorithm>
#include <cstring>

#include "launch.h"
#include "sigmakin_hs.cuh"

namespace mg {

// the currents kernel's own smaller CTA: 4 events, 128 threads, three CTAs per SM
template <class P, class R>
struct HsSplitA {
  using V = HsLane<P, R, CS_SIMT>;
  static constexpr int NT = 128, EV = 4, CTAS = 3, EW = LaneOf<V>::EW, EU = EV / EW;  // EU units
  static constexpr size_t o_proptab = 0;
  static constexpr size_t o_md = align_up(o_proptab + 8 * P::NPROP, 16);
  static constexpr size_t o_mconst = align_up(o_md + 16 * P::NMOM, 16);
  static constexpr size_t o_p = align_up(o_mconst + 32, 16);
  static constexpr size_t o_K = align_up(o_p + 8 * EV * P::NPAR * 4, 16);
  static constexpr size_t o_pr = align_up(o_K + sizeof(V) * EU * P::NMOM * 4, 16);
  static constexpr size_t o_cur = align_up(o_pr + 2 * sizeof(V) * EU * P::NPROP, 16);
  static constexpr size_t bytes = o_cur + sizeof(W4<V>) * EU * P::HS_NSLOT;
  static_assert(bytes <= 232448, "shared memory per CTA above the 227 KB limit");
};

template <class P, class R>
__global__ void __launch_bounds__(HsSplitA<P, R>::NT, HsSplitA<P, R>::CTAS)
    sigmakin_hs_currents_kernel(SigArgs a, Couplings<R> cp, int64_t first, int64_t last, uint4* __restrict__ rec) {
  using L = HsSplitA<P, R>;
  using V = typename L::V;
  using RC = HsRecord<P, V>;
  constexpr int NT = L::NT;
  extern __shared__ __align__(1024) unsigned char smem[];
  const int tid = threadIdx.x;
  const int64_t e0 = first + (int64_t)blockIdx.x * L::EV;
  if (e0 >= last) return;
  const int nev = (int)min((int64_t)L::EV, last - e0);
  uint4* curs = reinterpret_cast<uint4*>(smem + L::o_cur);
  hs_setup_words<P, R, L>(smem, a.pp);
  hs_load_momenta<P, R, L>(smem, a.mom, a.nevt, e0, nev);
  __syncthreads();
  const int nu = (nev + L::EW - 1) / L::EW;
  hs_tables<P, R, L, V>(smem, a.pp, nev, curs, cp);
  const V* Kall = reinterpret_cast<const V*>(smem + L::o_K);
  const cx<V>* prall = reinterpret_cast<const cx<V>*>(smem + L::o_pr);
  const Couplings<V> cv = lane_couplings<V>(cp);
  const HsItem* items = P::hs_items();
#pragma unroll
  for (int l = 1; l < P::HS_NLEVEL; ++l) {
    const int i0 = P::hs_level(l), ni = P::hs_level(l + 1) - i0, n = ni * nu;
    for (int t = tid; t < n; t += NT) {
      const int u = t / ni;
      const HsItem it = items[i0 + t - u * ni];
      const HsSlots<P, V, P::HS_NSLOT> cur{curs + u * RC::CUR};
      if constexpr (P::HS_ORDERED) ord_item<P, V>(it, cur, Kall + u * P::NMOM * 4, prall + u * P::NPROP, cv);
      else hs_item<P, V>(it, cur, Kall + u * P::NMOM * 4, prall + u * P::NPROP, cv);
    }
    __syncthreads();
  }
  const uint4* ks = reinterpret_cast<const uint4*>(smem + L::o_K);
  uint4* out = rec + (e0 - first) / L::EW * RC::WORDS;
  for (int t = tid; t < nu * RC::WORDS; t += NT) {
    const int u = t / RC::WORDS, w = t - u * RC::WORDS;
    if (w < RC::CUR + RC::KW) {
      out[t] = w < RC::CUR ? curs[u * RC::CUR + w] : ks[u * RC::KW + (w - RC::CUR)];
    } else {
      constexpr int PER = (int)(16 / sizeof(cx<V>));
      alignas(16) cx<V> f[PER];
#pragma unroll
      for (int k = 0; k < PER; ++k) {
        const int j = (w - RC::CUR - RC::KW) * PER + k;
        f[k] = prall[u * P::NPROP + min(j, P::NPROP - 1)];
      }
      out[t] = *reinterpret_cast<const uint4*>(f);
    }
  }
}

template <class P, class R>
__global__ void __launch_bounds__(HsCfg<P, R>::NT, HsCfg<P, R>::CTAS)
    sigmakin_hs_amplitudes_kernel(SigArgs a, Couplings<R> cp, int64_t first, int64_t last, const uint4* __restrict__ rec) {
  hs_sigmakin_body<P, R, CS_SIMT, kSrcRecords>(a, cp, first, last, rec);
}

template <class P, class R>
struct SplitLaunch {
  static cudaError_t prepare() {
    cudaError_t e = cudaFuncSetAttribute(sigmakin_hs_currents_kernel<P, R>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)HsSplitA<P, R>::bytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(sigmakin_hs_amplitudes_kernel<P, R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)HsLayout<P, R, CS_SIMT>::bytes);
  }
  static cudaError_t currents(const SigArgs& a, const Couplings<R>& cp, int64_t first, int64_t last, uint4* rec,
                              cudaStream_t s) {
    using L = HsSplitA<P, R>;
    const int64_t grid = (last - first + L::EV - 1) / L::EV;
    sigmakin_hs_currents_kernel<P, R><<<(unsigned)grid, L::NT, L::bytes, s>>>(a, cp, first, last, rec);
    return cudaGetLastError();
  }
  static cudaError_t amplitudes(const SigArgs& a, const Couplings<R>& cp, int64_t first, int64_t last,
                                const uint4* rec, cudaStream_t s) {
    using C = HsCfg<P, R>;
    int64_t grid = (last - first + C::EVMIN * C::EW - 1) / (C::EVMIN * C::EW);
    // a chunk of fewer full groups than SMs: over all of them (one unit per CTA at
    // least), as the single kernel's small batches (64 gg -> t t~ g events mixed 16.6 ->
    // 12.4 us, FP64 75 -> 60 us)
    int dev = 0, nsm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (grid < nsm) grid = std::min<int64_t>(nsm, (last - first + C::EW - 1) / C::EW);
    sigmakin_hs_amplitudes_kernel<P, R>
        <<<(unsigned)grid, C::NT, HsLayout<P, R, CS_SIMT>::bytes, s>>>(a, cp, first, last, rec);
    return cudaGetLastError();
  }
};

}  // namespace mg

namespace mg {

// bytes per event (a record holds the events of one lane)
template <class P, class R>
constexpr int64_t split_record_bytes() {
  using A = HsSplitA<P, R>;
  static_assert(HsRecord<P, typename A::V>::WORDS * 16 % A::EW == 0, "record in whole bytes per event");
  return (int64_t)HsRecord<P, typename A::V>::WORDS * 16 / A::EW;
}

// One batch through the split kernels: chunk = workspace / (2 records per event),
// a multiple of the currents kernel's events per CTA; the graph key holds every
// launch argument, so a call with other buffers or parameters re-captures.
template <class P, class R>
cudaError_t launch_split_impl(int proc, const SigLaunch& l, const Couplings<R>& cp, int mode, void* ws,
                              int64_t ws_bytes, cudaStream_t s) {
  constexpr int64_t rec_bytes = split_record_bytes<P, R>();
  int64_t chunk = ws_bytes / (2 * rec_bytes);
  // whole waves of the amplitudes kernel (all helicities good) where the
  // workspace allows: a partial last wave per chunk idles SMs
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return cudaGetLastError();
  const int64_t wave = (int64_t)nsm * HsCfg<P, R>::CTAS * HsCfg<P, R>::EVMIN * HsCfg<P, R>::EW;
  chunk -= chunk >= wave ? chunk % wave : chunk % HsSplitA<P, R>::EV;
  if (chunk < HsSplitA<P, R>::EV) return cudaErrorInvalidValue;
  if (l.nevt == 0) return cudaSuccess;
  if (chunk > l.nevt) chunk = (l.nevt + HsSplitA<P, R>::EV - 1) / HsSplitA<P, R>::EV * HsSplitA<P, R>::EV;
  struct Key {
    int proc_mode;
    int device;  // a graph belongs to the device it was captured on
    SigArgs a;
    Couplings<R> cp;
    void* ws;
    int64_t chunk;
  } key;
  std::memset(static_cast<void*>(&key), 0, sizeof key);  // padding compared too: members set one by one
  key.proc_mode = proc * 16 + mode;
  key.device = dev;
  key.a.nevt = l.nevt;
  key.a.mom = l.mom;
  key.a.mask = l.mask;
  key.a.me = l.me;
  key.a.pp = l.pp;
  key.a.hel_rnd = l.hel_rnd;
  key.a.hel_out = l.hel_out;
  key.a.col_rnd = l.col_rnd;
  key.a.col_out = l.col_out;
  key.cp = cp;
  key.ws = ws;
  key.chunk = chunk;
  const SigArgs a = key.a;
  SplitOps ops;
  ops.prepare = [] { return SplitLaunch<P, R>::prepare(); };
  ops.currents = [a, cp](int64_t f, int64_t e, void* rec, cudaStream_t st) {
    return SplitLaunch<P, R>::currents(a, cp, f, e, static_cast<uint4*>(rec), st);
  };
  ops.amplitudes = [a, cp](int64_t f, int64_t e, const void* rec, cudaStream_t st) {
    return SplitLaunch<P, R>::amplitudes(a, cp, f, e, static_cast<const uint4*>(rec), st);
  };
  char* b0 = static_cast<char*>(ws);
  return run_split_graph(&key, sizeof key, l.nevt, chunk, b0, b0 + chunk * rec_bytes, ops, s);
}

}  // namespace mg

// One translation unit per process and precision (they compile in parallel):
// MG_DEFINE_SPLIT_LAUNCHERS with the FP32 kernels and the dispatcher,
// MG_INSTANTIATE_SPLIT_FP64 with the FP64 kernels.
#define MG_DEFINE_SPLIT_LAUNCHERS(N)                                                                    \
  namespace mg {                                                                                         \
  extern template cudaError_t launch_split_impl<Proc##N, double>(int, const SigLaunch&,                 \
                                                                  const Couplings<double>&, int, void*, \
                                                                  int64_t, cudaStream_t);               \
  int64_t split_record_bytes_p##N(int mode) {                                                           \
    return mode == 0 ? split_record_bytes<Proc##N, double>()                                            \
                     : split_record_bytes<Proc##N, float>();                                             \
  }                                                                                                      \
  cudaError_t launch_sigmakin_split_p##N(const SigLaunch& l, int mode, void* ws, int64_t ws_bytes,      \
                                         cudaStream_t s) {                                               \
    if (mode == 0) return launch_split_impl<Proc##N, double>(N, l, l.cd, mode, ws, ws_bytes, s);         \
    if (mode == 2) return launch_split_impl<Proc##N, float>(N, l, l.cf, mode, ws, ws_bytes, s);          \
    return cudaErrorInvalidValue;                                                                        \
  }                                                                                                      \
  }

#define MG_INSTANTIATE_SPLIT_FP64(N)                                                                    \
  namespace mg {                                                                                         \
  template cudaError_t launch_split_impl<Proc##N, double>(int, const SigLaunch&, const Couplings<double>&, \
                                                          int, void*, int64_t, cudaStream_t);           \
  }
