// dwf_launch.cuh -- host-side launchers of the kernel templates, instantiated once per
// precision in k_f64.cu / k_f32.cu / k_half.cu so the three compile in parallel.
#pragma once

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <tuple>

#include "dwf_kernels.cuh"
#include "dwf_optin.h"

namespace dwf {

// threads per CTA of the per-site kernels: the Ns slices of spb sites, about 128
// (at most 64 sites, which bounds the shared memory of small-Ns CTAs)
inline int sites_per_block(int Ns) {
  int spb = 128 / Ns;
  if (spb > 64) spb = 64;
  return spb < 1 ? 1 : spb;
}

// sites per CTA of k_hop, whose CTA is (Ns, spb): 128 threads measured best at Ns = 16
// (against 256 and 512 threads, and 64 and 96, for the FP32 hop kernels); in FP64 at most 62
// sites, of whose links (1168 bytes each) three CTAs fit on an SM
inline int hop_sites_per_block(int P, int Ns) {
  const int target = 128, most = P == P_F64 ? 62 : 64;
  int spb = target / Ns;
  if (spb > most) spb = most;
  return spb < 1 ? 1 : spb;
}

inline int vec_grid(long n, int sm_count) {
  long g = (n + 255) / 256;
  long cap = (long)sm_count * 8;
  if (g > cap) g = cap;
  return (int)(g < 1 ? 1 : g);
}

// a launch, overlapping its predecessor's end if pdl (see pdl_wait)
template <typename... A, typename... B>
cudaError_t launch(void (*k)(A...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl, const B &...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, A(args)...);
}

// allows kernel k `smem` bytes of dynamic shared memory on the current device
template <typename... A>
cudaError_t allow_smem(SmemOptIn &seen, void (*k)(A...), size_t smem) {
  if (smem <= kSmemNoOptIn) return cudaSuccess;
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  return (cudaError_t)seen.ensure(dev, smem, [&] {
    return (int)cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  });
}

template <int P, int EPI, int NSC>
cudaError_t hop_go(const HopArgs &a, cudaStream_t st) {
  // the shape the host chose (autotuner), else 128-thread CTAs, persistent without M5 (not FP64)
  int spb = hop_sites_per_block(P, a.Ns);
  bool persistent = hop_persistent<P, EPI>();
  if (a.shape_threads > 0) {
    spb = std::max(1, std::min(64, a.shape_threads / a.Ns));
    persistent = a.shape_persistent != 0;
  }
  if (spb * a.Ns > 256) return cudaErrorInvalidConfiguration;
  const size_t smem = hop_smem_bytes<P, EPI>(spb, a.Ns);
  static SmemOptIn optin;
  cudaError_t e = allow_smem(optin, k_hop<P, EPI, NSC>, smem);
  if (e != cudaSuccess) return e;
  const int nrhs = a.nrhs > 1 ? a.nrhs : 1;
  const long ntile = (a.h + spb - 1) / spb;
  long nblk = ntile;  // one tile per CTA
  if (persistent) {
    // persistent grid: as many CTAs per right-hand side as are resident at once, each taking
    // an equal number of tiles (the rows of a batch follow one another through the GPU, and
    // a finished right-hand side's row returns at once)
    const int nthr = a.Ns * spb;
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    // resident CTAs per GPU for this kernel, CTA size and shared memory (cached)
    static std::mutex mu;
    static std::map<std::tuple<int, int, size_t>, long> resident;
    const auto key = std::make_tuple(dev, nthr, smem);
    long res = 0;
    {
      std::lock_guard<std::mutex> lock(mu);
      auto it = resident.find(key);
      if (it != resident.end()) res = it->second;
    }
    if (res <= 0) {
      int sms = 0, per = 0;
      e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_hop<P, EPI, NSC>, nthr, smem);
      if (e != cudaSuccess) return e;
      res = (long)std::max(per, 1) * sms;
      std::lock_guard<std::mutex> lock(mu);
      resident[key] = res;
    }
    const long per_cta = (ntile + res - 1) / res;
    nblk = (ntile + per_cta - 1) / per_cta;
  }
  return launch(k_hop<P, EPI, NSC>, dim3((unsigned)nblk, nrhs), dim3(a.Ns, spb), smem, st, a.pdl, a);
}

// the inner CG's kernels and those of C get a compile-time Ns for the fifth-dimension extents in
// use (C's second hop at 16^3x32x16: 126 registers and 124 us with Ns at run time)
template <int P, int EPI>
cudaError_t hop_ns(const HopArgs &a, cudaStream_t st) {
  if constexpr (P != P_F64 && (EPI == E_M || EPI == E_XPAY_G5 || EPI == E_CG_UPDATE || EPI == E_M_XPAY)) {
    switch (a.Ns) {
      case 8: return hop_go<P, EPI, 8>(a, st);
      case 12: return hop_go<P, EPI, 12>(a, st);
      case 16: return hop_go<P, EPI, 16>(a, st);
      case 20: return hop_go<P, EPI, 20>(a, st);
      case 24: return hop_go<P, EPI, 24>(a, st);
      case 32: return hop_go<P, EPI, 32>(a, st);
      default: break;
    }
  }
  return hop_go<P, EPI, 0>(a, st);
}

template <int P>
cudaError_t hop_launch(int epi, const HopArgs &a, cudaStream_t st) {
  switch (epi) {
    case E_PLAIN: return hop_ns<P, E_PLAIN>(a, st);
    case E_M: return hop_ns<P, E_M>(a, st);
    case E_XPAY_G5: return hop_ns<P, E_XPAY_G5>(a, st);
    case E_XPAY: return hop_ns<P, E_XPAY>(a, st);
    case E_M_XPAY: return hop_ns<P, E_M_XPAY>(a, st);
    case E_CG_UPDATE: return hop_ns<P, E_CG_UPDATE>(a, st);
    case E_RESID: return hop_ns<P, E_RESID>(a, st);
  }
  return cudaErrorInvalidValue;
}

// sites per CTA of k_smix.  CTAs of about 128 threads for small and middle Ns: the p-update's three
// operands in flight take 88 registers, five CTAs per SM (4^4x8: 31.2 -> 29.4 us an iteration, 12
// rows of 8^4x8: 77.1 -> 75.2 ms a solve).  Every CTA stages the matrices, 2 Ns^2 reals (S_DUAL
// 4), which at large Ns cost more than its sites: there 256 threads, so twice the sites.  128 and
// 256 threads on 12^3x16 in FP32: D at Ns = 28 317 and 316 us, 32 331 and 326, 48 630 and 538, 64
// 1005 and 808; M5 at 32 118 and 118.5, 33 140 and 137, 64 268 and 256; an iteration at 32 227 and
// 230, 40 366 and 368, 48 459 and 460 (bf16 500 and 492), 64 650 and 631.
inline int smix_sites_per_block(int P, int mode, int Ns) {
  const int wide_from = mode == S_DUAL ? 32 : mode == S_CGP ? 48 : 33;
  return P != P_F64 && Ns >= wide_from ? 256 / Ns : sites_per_block(Ns);
}

template <int P, int MODE>
cudaError_t smix_go(const SmixArgs &a, cudaStream_t st) {
  const int spb = smix_sites_per_block(P, MODE, a.Ns);
  const size_t smem = smix_smem_bytes<P>(spb, a.Ns, MODE == S_DUAL);
  static SmemOptIn optin;
  const cudaError_t e = allow_smem(optin, k_smix<P, MODE>, smem);
  if (e != cudaSuccess) return e;
  const long nblk = (a.h + spb - 1) / spb;
  return launch(k_smix<P, MODE>, dim3((unsigned)nblk, a.nrhs > 1 ? a.nrhs : 1), dim3(a.Ns, spb), smem, st, a.pdl, a);
}

// FP64 recurrences: CTAs of about 128 threads, so that several share an SM and one's loads
// overlap another's FP64 phase (at most 37 KB of shared memory, at Ns = 2)
template <int MODE>
cudaError_t srec_go(const SmixArgs &a, cudaStream_t st) {
  const int spb = sites_per_block(a.Ns);
  const size_t smem = srec_smem_bytes(spb, a.Ns);
  const long nblk = (a.h + spb - 1) / spb;
  return launch(k_srec<MODE>, dim3((unsigned)nblk, a.nrhs > 1 ? a.nrhs : 1), dim3(a.Ns, spb), smem, st, a.pdl, a);
}

cudaError_t sdual_launch(const SmixArgs &a, cudaStream_t st);

template <int P>
cudaError_t smix_launch(int mode, const SmixArgs &a, cudaStream_t st) {
  if constexpr (P == P_F64) {
    // as recurrences; dense only where a matrix has no table as accurate as its rows (16^3x32x16:
    // 210 us against 693 us)
    switch (mode) {
      case S_PLAIN: return a.rec ? srec_go<S_PLAIN>(a, st) : smix_go<P, S_PLAIN>(a, st);
      case S_G5: return a.rec ? srec_go<S_G5>(a, st) : smix_go<P, S_G5>(a, st);
      case S_CGP: return a.rec ? srec_go<S_CGP>(a, st) : smix_go<P, S_CGP>(a, st);
      case S_DUAL: return sdual_launch(a, st);
    }
  } else {
    switch (mode) {
      case S_PLAIN: return smix_go<P, S_PLAIN>(a, st);
      case S_G5: return smix_go<P, S_G5>(a, st);
      case S_CGP: return smix_go<P, S_CGP>(a, st);
      case S_DUAL: return smix_go<P, S_DUAL>(a, st);
    }
  }
  return cudaErrorInvalidValue;
}

template <int P>
cudaError_t norm2_launch(const VecArgs &v, int sm_count, cudaStream_t st) {
  k_norm2<P><<<vec_grid(v.n, sm_count), 256, 0, st>>>(v);
  return cudaGetLastError();
}

template <int PA, int PB>
cudaError_t convert_go(const VecArgs &v, int sm_count, cudaStream_t st) {
  k_convert<PA, PB><<<vec_grid(v.n, sm_count), 256, 0, st>>>(v);
  return cudaGetLastError();
}

// conversions between FP64 and precision P, both directions
template <int P>
cudaError_t convert_launch(int to_p, const VecArgs &v, int sm_count, cudaStream_t st) {
  if (to_p) return convert_go<P_F64, P>(v, sm_count, st);
  return convert_go<P, P_F64>(v, sm_count, st);
}

template <int P>
cudaError_t accum_launch(const VecArgs &v, int sm_count, cudaStream_t st) {
  k_accum<P><<<vec_grid(v.n, sm_count), 256, 0, st>>>(v);
  return cudaGetLastError();
}

template <int P>
cudaError_t pack_launch(const double *host, Field out, Geom g, int parity, cudaStream_t st) {
  const int spb = sites_per_block(g.Ns);
  k_pack<P><<<(unsigned)((g.h + spb - 1) / spb), dim3(g.Ns, spb), host_stage_bytes(spb, g.Ns), st>>>(host, out, g, parity);
  return cudaGetLastError();
}

template <int P>
cudaError_t unpack_launch(Field in, double *host, Geom g, int parity, int zero_other, cudaStream_t st) {
  const int spb = sites_per_block(g.Ns);
  return launch(k_unpack<P>, dim3((unsigned)((g.h + spb - 1) / spb)), dim3(g.Ns, spb), host_stage_bytes(spb, g.Ns), st, true,
                in, host, g, parity, zero_other);
}

template <int P>
cudaError_t gauge_launch(const double *U, void *G, Geom g, int parity, int sm_count, cudaStream_t st) {
  k_gauge<P><<<vec_grid(g.h * 8, sm_count), 256, 0, st>>>(U, static_cast<typename PT<P>::lreal *>(G), g,
                                                            parity);
  return cudaGetLastError();
}

// one set of entry points per precision
#define DWF_DECLARE_PREC(P)                                                                           \
  extern template cudaError_t hop_launch<P>(int, const HopArgs &, cudaStream_t);                     \
  extern template cudaError_t smix_launch<P>(int, const SmixArgs &, cudaStream_t);                   \
  extern template cudaError_t norm2_launch<P>(const VecArgs &, int, cudaStream_t);                   \
  extern template cudaError_t convert_launch<P>(int, const VecArgs &, int, cudaStream_t);            \
  extern template cudaError_t accum_launch<P>(const VecArgs &, int, cudaStream_t);                   \
  extern template cudaError_t pack_launch<P>(const double *, Field, Geom, int, cudaStream_t);         \
  extern template cudaError_t unpack_launch<P>(Field, double *, Geom, int, int, cudaStream_t);       \
  extern template cudaError_t gauge_launch<P>(const double *, void *, Geom, int, int, cudaStream_t);

#define DWF_INSTANTIATE_PREC(P)                                                                \
  template cudaError_t hop_launch<P>(int, const HopArgs &, cudaStream_t);                     \
  template cudaError_t smix_launch<P>(int, const SmixArgs &, cudaStream_t);                   \
  template cudaError_t norm2_launch<P>(const VecArgs &, int, cudaStream_t);                   \
  template cudaError_t convert_launch<P>(int, const VecArgs &, int, cudaStream_t);            \
  template cudaError_t accum_launch<P>(const VecArgs &, int, cudaStream_t);                   \
  template cudaError_t pack_launch<P>(const double *, Field, Geom, int, cudaStream_t);         \
  template cudaError_t unpack_launch<P>(Field, double *, Geom, int, int, cudaStream_t);       \
  template cudaError_t gauge_launch<P>(const double *, void *, Geom, int, int, cudaStream_t);

#ifndef DWF_KERNEL_TU
DWF_DECLARE_PREC(P_F64)
DWF_DECLARE_PREC(P_F32)
DWF_DECLARE_PREC(P_F16)
DWF_DECLARE_PREC(P_BF16)
#endif

cudaError_t neighbours_launch(int *nbr, Geom g, int parity, int sm_count, cudaStream_t st);
cudaError_t diff_norm2_launch(const VecArgs &v, int sm_count, cudaStream_t st);
cudaError_t host_axpy_launch(const HostAxpyArgs &v, int sm_count, cudaStream_t st);
cudaError_t point_sources_launch(double *rhs, long x0site, long V4, int Ns, cudaStream_t st);
cudaError_t prop_extract_launch(const double *sol, double *prop, long V4, int Ns, int sm_count, cudaStream_t st);

}  // namespace dwf
