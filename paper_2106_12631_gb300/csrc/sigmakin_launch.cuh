// Launchers shared by the per-process translation units (one TU per process
// so the four diagram programs compile in parallel).
#pragma once
#include <atomic>

#include "launch.h"
#include "sigmakin.cuh"
#include "sigmakin_hs.cuh"

namespace mg {

template <class P, class R, int CS>
cudaError_t launch_sigmakin_variant(const SigArgs& a, const Couplings<R>& cp, int64_t grid, cudaStream_t s) {
  using L = SigLayout<P, R, CS>;
  auto k = sigmakin_kernel<P, R, CS>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes);
  if (e != cudaSuccess) return e;
  k<<<(unsigned)grid, SigCfg<P>::NT, L::bytes, s>>>(a, cp);
  return cudaGetLastError();
}

// The helicity-shared kernel runs persistent: as many CTAs as are resident at
// once (SMs x CTAs per SM, cached per device), each looping over groups of
// events (the CTA's group count follows from the mask and the grid on the device;
// a batch that does not fill the CTAs is spread over all of them).  CTAs
// per SM: the larger of the occupancy query and the count the kernel's shared
// memory budget and launch bounds are built for (the query has returned 1 for
// the tcgen05 variant, whose two CTAs per SM fit); should fewer fit, the
// surplus CTAs start later and take their groups then.
// ra != nullptr: the kernel that runs RAMBO itself (sigmakin_hs_rambo_kernel).
template <class P, class R, int CS, bool FUSED = false>
cudaError_t launch_sigmakin_hs_variant(const SigArgs& a, const Couplings<R>& cp, int64_t grid, cudaStream_t s,
                                       const RamboArgs* ra = nullptr) {
  using L = HsLayout<P, R, CS, FUSED>;
  using H = typename L::H;
  constexpr int NT = L::NT;
  constexpr int kMaxDevices = 64;
  struct Fit {
    int cap, per;  // CTAs resident on the whole device and per SM; 0 until known
  };
  static std::atomic<Fit> resident[kMaxDevices];
  const void* k = FUSED ? (const void*)sigmakin_hs_rambo_kernel<P, R, CS> : (const void*)sigmakin_hs_kernel<P, R, CS>;
  // A batch that one round of k CTAs per SM holds (all helicities good) takes the
  // k that leaves the fewest events to an SM, and of two such the smaller (1000
  // events of 8 per CTA on 152 SMs of two CTAs: one CTA of 7, not two of 4; a
  // grid of all CTAs with idle ones would put the busy ones side by side).  Choices
  // take one warp per event: in the mixed mode, which waits for them, first the k
  // with the fewest rounds of the CTA's warps (2001 gg -> t t~ events 14.6 -> 11.7
  // us; FP64, bound by its pipe, 2432 events 29.3 us, by rounds 32.0).
  auto launch = [&](Fit f) {
    const int64_t nsm = f.cap / f.per, units = (a.nevt + H::EW - 1) / H::EW;
    const bool choices = sizeof(R) == 4 && (a.hel_out || a.col_out);
    int64_t g = f.cap, load = INT64_MAX;
    for (int k = 1; k <= f.per; ++k) {
      const int64_t u = (units + nsm * k - 1) / (nsm * k);
      const int64_t rounds = choices ? (u * H::EW + NT / 32 - 1) / (NT / 32) : 0;
      if (u <= H::EVMIN && (rounds << 32) + u * k < load) {
        g = nsm * k;
        load = (rounds << 32) + u * k;
      }
    }
    if (g > units) g = units;  // one unit per CTA at least
    // the launch's own status, not the thread's last error: that may be an
    // earlier call's, which is not ours to answer with a second launch
    void* args[] = {const_cast<SigArgs*>(&a), const_cast<Couplings<R>*>(&cp), const_cast<RamboArgs*>(ra)};
    const cudaError_t e = cudaLaunchKernel(k, dim3((unsigned)g), dim3(NT), args, L::bytes, s);
    if (e != cudaSuccess) cudaGetLastError();  // reported by the return value
    return e;
  };
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  Fit fit = dev < kMaxDevices ? resident[dev].load(std::memory_order_relaxed) : Fit{0, 0};
  // the shared-memory attribute is set with the first launch on a device, and
  // again if a launch is refused for want of it (the device was reset)
  if (fit.cap != 0 && (e = launch(fit)) != cudaErrorInvalidValue) return e;
  if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes)) != cudaSuccess) return e;
  int nsm = 0, per = 0;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, NT, L::bytes)) != cudaSuccess) return e;
  if (per < H::CTAS) per = H::CTAS;
  fit = Fit{nsm * per, per};
  if (dev < kMaxDevices) resident[dev].store(fit, std::memory_order_relaxed);
  return launch(fit);
}

// mode 0 FP64; 1 mixed, colour sum on CUDA cores below 48 colour flows and on
// the tensor cores from 48 on; 2 mixed + CUDA-core colour sum; 5 mixed +
// tcgen05 colour sum (helicity-shared kernel); 3 FP64, 4 mixed + tcgen05 with
// the per-helicity unrolled kernel (every helicity recomputes all its currents)
inline SigArgs sig_args(const SigLaunch& l) {
  return SigArgs{l.nevt, l.mom, l.mask, l.me, l.mask_out, l.pp, l.hel_rnd, l.hel_out, l.col_rnd, l.col_out};
}

template <class P>
cudaError_t launch_sigmakin_impl(const SigLaunch& l, int mode, cudaStream_t s) {
  const SigArgs a = sig_args(l);
  const int64_t grid = (l.nevt + SigCfg<P>::EVMIN - 1) / SigCfg<P>::EVMIN;
  if (grid == 0) return cudaSuccess;
  constexpr bool tc_default = P::NCOLOR >= 48;
  switch (mode) {
    case 0: return launch_sigmakin_hs_variant<P, double, CS_SIMT>(a, l.cd, grid, s);
    case 1:
      return tc_default ? launch_sigmakin_hs_variant<P, float, CS_TC>(a, l.cf, grid, s)
                        : launch_sigmakin_hs_variant<P, float, CS_SIMT>(a, l.cf, grid, s);
    case 2: return launch_sigmakin_hs_variant<P, float, CS_SIMT>(a, l.cf, grid, s);
    case 5: return launch_sigmakin_hs_variant<P, float, CS_TC>(a, l.cf, grid, s);
    case 3: return launch_sigmakin_variant<P, double, CS_SIMT>(a, l.cd, grid, s);
    case 4: return launch_sigmakin_variant<P, float, CS_TC>(a, l.cf, grid, s);
  }
  return cudaErrorInvalidValue;
}

// RAMBO and SIGMAKIN in one kernel; the helicity-shared modes only (0 FP64,
// 1 mixed, 2 mixed + CUDA-core colour sum, 5 mixed + tcgen05 colour sum)
template <class P>
cudaError_t launch_sigmakin_rambo_impl(const SigLaunch& l, int mode, cudaStream_t s) {
  const SigArgs a = sig_args(l);
  const RamboArgs ra{l.rnd, l.wgt, l.ecm, l.key, l.first_event, l.st};
  if (l.nevt == 0) return cudaSuccess;
  constexpr bool tc_default = P::NCOLOR >= 48;
  switch (mode) {
    case 0: return launch_sigmakin_hs_variant<P, double, CS_SIMT, true>(a, l.cd, 0, s, &ra);
    case 1:
      return tc_default ? launch_sigmakin_hs_variant<P, float, CS_TC, true>(a, l.cf, 0, s, &ra)
                        : launch_sigmakin_hs_variant<P, float, CS_SIMT, true>(a, l.cf, 0, s, &ra);
    case 2: return launch_sigmakin_hs_variant<P, float, CS_SIMT, true>(a, l.cf, 0, s, &ra);
    case 5: return launch_sigmakin_hs_variant<P, float, CS_TC, true>(a, l.cf, 0, s, &ra);
  }
  return cudaErrorInvalidValue;
}

template <class P>
cudaError_t launch_filter_impl(const SigLaunch& l, cudaStream_t s) {
  using L = SigLayout<P, double, CS_SIMT>;
  SigArgs a{l.nevt, l.mom, l.mask, l.me, l.mask_out, l.pp, nullptr, nullptr};
  const int64_t grid = l.nevt * ((P::NHEL + FILTER_NT - 1) / FILTER_NT);
  if (grid == 0) return cudaSuccess;
  auto k = filter_kernel<P>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes);
  if (e != cudaSuccess) return e;
  k<<<(unsigned)grid, FILTER_NT, L::bytes, s>>>(a, l.cd);
  return cudaGetLastError();
}

}  // namespace mg

// The FP64 kernels of a process (sum and filter) are instantiated in their own
// translation unit (MG_INSTANTIATE_FP64), the FP32 ones with the dispatcher.
#define MG_DEFINE_PROCESS_LAUNCHERS(N)                                                                  \
  namespace mg {                                                                                         \
  extern template cudaError_t launch_sigmakin_variant<Proc##N, double, CS_SIMT>(                        \
      const SigArgs&, const Couplings<double>&, int64_t, cudaStream_t);                                  \
  extern template cudaError_t launch_sigmakin_hs_variant<Proc##N, double, CS_SIMT>(                     \
      const SigArgs&, const Couplings<double>&, int64_t, cudaStream_t, const RamboArgs*);                \
  extern template cudaError_t launch_sigmakin_hs_variant<Proc##N, double, CS_SIMT, true>(               \
      const SigArgs&, const Couplings<double>&, int64_t, cudaStream_t, const RamboArgs*);                \
  extern template cudaError_t launch_filter_impl<Proc##N>(const SigLaunch&, cudaStream_t);              \
  cudaError_t launch_sigmakin_p##N(const SigLaunch& a, int mode, cudaStream_t s) {                      \
    return launch_sigmakin_impl<Proc##N>(a, mode, s);                                                    \
  }                                                                                                      \
  cudaError_t launch_sigmakin_rambo_p##N(const SigLaunch& a, int mode, cudaStream_t s) {                \
    return launch_sigmakin_rambo_impl<Proc##N>(a, mode, s);                                              \
  }                                                                                                      \
  cudaError_t launch_filter_p##N(const SigLaunch& a, cudaStream_t s) { return launch_filter_impl<Proc##N>(a, s); } \
  }

#define MG_INSTANTIATE_FP64(N)                                                                          \
  namespace mg {                                                                                         \
  template cudaError_t launch_sigmakin_variant<Proc##N, double, CS_SIMT>(                               \
      const SigArgs&, const Couplings<double>&, int64_t, cudaStream_t);                                  \
  template cudaError_t launch_sigmakin_hs_variant<Proc##N, double, CS_SIMT>(                            \
      const SigArgs&, const Couplings<double>&, int64_t, cudaStream_t, const RamboArgs*);                \
  template cudaError_t launch_sigmakin_hs_variant<Proc##N, double, CS_SIMT, true>(                      \
      const SigArgs&, const Couplings<double>&, int64_t, cudaStream_t, const RamboArgs*);                \
  template cudaError_t launch_filter_impl<Proc##N>(const SigLaunch&, cudaStream_t);                     \
  }
