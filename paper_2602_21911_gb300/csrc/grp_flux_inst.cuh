// Launchers of the flux and persistent batched kernels for one system, degree
// and reconstruction, defined by macro so that each (degree, reconstruction)
// instantiation sits in a translation unit of its own and they compile in
// parallel.  gamma = 7/5 takes the fast-path instantiation.
#pragma once
#include "grp_kernels.cuh"
#include "grp_launch.h"

namespace grp {
// the first pass in fixed point, where the caller chose it (flux_fixed)
template <int MM, bool NLV>
inline bool launch_flux_fixed(const StepArgs& a, cudaStream_t s)
{
  if (!a.fixed) return false;
  const unsigned tpb = spread(a.nif, 128);
  if constexpr (!NLV) {
    k_flux_fixed<MM><<<(unsigned)((a.nif + tpb - 1) / tpb), tpb, 0, s>>>(a);
  }
  else if constexpr (MM <= 3) k_flux_fixed_nl<MM><<<(unsigned)((flux_threads(a.nif) + tpb - 1) / tpb), tpb, 0, s>>>(a);
  return true;
}

// the second pass, where the first leaves it interfaces
template <int MM, bool NLV>
inline void launch_flux_hard(const StepArgs& a, cudaStream_t s)
{
  constexpr bool DEFER = flux_defers_at<SYS_EULER, MM, NLV, false>();
  if constexpr (!NLV || MM <= 3) {
    if (a.hard_cap > 0 && (DEFER || a.fixed)) {
      static int sms[64] = {0};
      int dev = 0;
      cudaGetDevice(&dev);
      if (dev < 0 || dev >= 64) dev = 0;
      if (!sms[dev]) cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev);
      const unsigned gh = hard_blocks(a.hard_cap, sms[dev] > 0 ? sms[dev] : 1);
      if constexpr (DEFER) {
        const bool net = flux_hard_net(a);
        if (a.ph.gamma == 1.4) {
          if (net) k_flux_hard<MM, true, true><<<gh, GRP_HARD_TPB, 0, s>>>(a);
          else k_flux_hard<MM, true, false><<<gh, GRP_HARD_TPB, 0, s>>>(a);
        } else {
          if (net) k_flux_hard<MM, false, true><<<gh, GRP_HARD_TPB, 0, s>>>(a);
          else k_flux_hard<MM, false, false><<<gh, GRP_HARD_TPB, 0, s>>>(a);
        }
      } else {
        k_flux_hard<MM, true, false, NLV><<<gh, GRP_HARD_TPB, 0, s>>>(a);      // gamma = 7/5 only
      }
    }
  }
}
}  // namespace grp

#define GRP_DEFINE_EULER_LAUNCHERS(MM, NLV, SUFFIX)                                                          \
  cudaError_t launch_flux_euler_##SUFFIX(const StepArgs& a, cudaStream_t s)                                  \
  {                                                                                                          \
    const unsigned tpb = spread(a.nif, GRP_FLUX_TPB), g = (unsigned)((flux_threads(a.nif) + tpb - 1) / tpb); \
    if (launch_flux_fixed<MM, NLV>(a, s)) {}                                                                 \
    else if (a.ph.gamma == 1.4) k_flux<SYS_EULER, MM, true, NLV><<<g, tpb, 0, s>>>(a);              \
    else k_flux<SYS_EULER, MM, false, NLV><<<g, tpb, 0, s>>>(a);                                    \
    launch_flux_hard<MM, NLV>(a, s);                                                                         \
    return cudaGetLastError();                                                                               \
  }                                                                                                          \
  cudaError_t launch_batch_euler_##SUFFIX(const BatchLaunch& L, cudaStream_t s)                              \
  {                                                                                                          \
    if (L.a.ph.gamma == 1.4)                                                                                 \
      k_batch<SYS_EULER, MM, true, NLV><<<L.blocks, L.threads, 0, s>>>(L.a, L.grp, L.nsteps, L.parity, L.A0, \
                                                                       L.A1, L.I0, L.I1);                    \
    else                                                                                                     \
      k_batch<SYS_EULER, MM, false, NLV><<<L.blocks, L.threads, 0, s>>>(L.a, L.grp, L.nsteps, L.parity,      \
                                                                        L.A0, L.A1, L.I0, L.I1);             \
    return cudaGetLastError();                                                                               \
  }

#define GRP_DEFINE_ADV_LAUNCHERS(NLV, SUFFIX)                                                                \
  cudaError_t launch_flux_adv##SUFFIX(const StepArgs& a, cudaStream_t s)                                     \
  {                                                                                                          \
    const unsigned tpb = spread(a.nif, GRP_FLUX_TPB), g = (unsigned)((flux_threads(a.nif) + tpb - 1) / tpb); \
    switch (a.M) {                                                                                           \
      case 1: k_flux<SYS_ADV, 1, false, NLV><<<g, tpb, 0, s>>>(a); break;                                    \
      case 2: k_flux<SYS_ADV, 2, false, NLV><<<g, tpb, 0, s>>>(a); break;                                    \
      case 3: k_flux<SYS_ADV, 3, false, NLV><<<g, tpb, 0, s>>>(a); break;                                    \
      case 4: k_flux<SYS_ADV, 4, false, NLV><<<g, tpb, 0, s>>>(a); break;                                    \
      default: return cudaErrorInvalidValue;                                                                 \
    }                                                                                                        \
    return cudaGetLastError();                                                                               \
  }                                                                                                          \
  cudaError_t launch_adv_step##SUFFIX(const StepArgs& a, DomStep* next, cudaStream_t s)                      \
  {                                                                                                          \
    const unsigned tpb = spread(a.ncell, 256), g = (unsigned)((a.ncell + tpb - 1) / tpb);                    \
    switch (a.M) {                                                                                           \
      case 1: k_adv_step<1, NLV><<<g, tpb, 0, s>>>(a, next); break;                                          \
      case 2: k_adv_step<2, NLV><<<g, tpb, 0, s>>>(a, next); break;                                          \
      case 3: k_adv_step<3, NLV><<<g, tpb, 0, s>>>(a, next); break;                                          \
      case 4: k_adv_step<4, NLV><<<g, tpb, 0, s>>>(a, next); break;                                          \
      default: return cudaErrorInvalidValue;                                                                 \
    }                                                                                                        \
    return cudaGetLastError();                                                                               \
  }                                                                                                          \
  cudaError_t launch_batch_adv##SUFFIX(const BatchLaunch& L, cudaStream_t s)                                 \
  {                                                                                                          \
    switch (L.a.M) {                                                                                         \
      case 1: k_batch<SYS_ADV, 1, false, NLV><<<L.blocks, L.threads, 0, s>>>(L.a, L.grp, L.nsteps, L.parity, \
                                                                             L.A0, L.A1, L.I0, L.I1); break; \
      case 2: k_batch<SYS_ADV, 2, false, NLV><<<L.blocks, L.threads, 0, s>>>(L.a, L.grp, L.nsteps, L.parity, \
                                                                             L.A0, L.A1, L.I0, L.I1); break; \
      case 3: k_batch<SYS_ADV, 3, false, NLV><<<L.blocks, L.threads, 0, s>>>(L.a, L.grp, L.nsteps, L.parity, \
                                                                             L.A0, L.A1, L.I0, L.I1); break; \
      case 4: k_batch<SYS_ADV, 4, false, NLV><<<L.blocks, L.threads, 0, s>>>(L.a, L.grp, L.nsteps, L.parity, \
                                                                             L.A0, L.A1, L.I0, L.I1); break; \
      default: return cudaErrorInvalidValue;                                                                 \
    }                                                                                                        \
    return cudaGetLastError();                                                                               \
  }
