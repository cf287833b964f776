// dwf_device.cuh -- device code of the domain-wall solver for sm_103a.
//
// Data layout in HBM (one parity of the 4D lattice at a time; cb = checkerboard index of
// a site within its parity, cb = site / 2 with site = x + Nx (y + Ny (z + Nz t))):
//   spinor (Sec. 3.1 "Vector Index Conversion", re-derived for 16-byte loads):
//     chunk k of (cb, s) at element ((cb * NCH + k) * Ns + s) of 16-byte chunks, so the
//     Ns threads of one site read consecutive 16 bytes for every chunk;
//     F64: 12 chunks of double2, F32: 6 chunks of float4, F16/BF16: 3 chunks of 8
//     halves plus a per-(cb, s) FP32 norm at nrm[cb * Ns + s].
//     Inside a (cb, s) the 24 reals keep the host order c = reim + 2 (colour + 3 spin).
//   gauge, doubled per output parity: G[p][cb][dir][*] with dir 0..3 = U_mu(x) and
//     dir 4..7 = U_mu(x - mu)^dagger (stored daggered), 18 reals (F64/F32) or the first
//     two rows, 12 reals (F16/BF16; the third row is rebuilt as conj(row0 x row1)).
//   neighbours: nbr[p][cb][dir] = cb of x + mu (dir < 4) / x - mu (dir >= 4) in parity 1-p.
//
// The hopping term of Eq. 12 is evaluated as H = sum_mu [(1 - g_mu) U psi(x+mu) +
// (1 + g_mu) U^dag psi(x-mu)] with D = -H/2.  In the chiral basis g_mu = [[0, A],[A^dag, 0]]
// so (1 + S g_mu) psi = (h, S A^dag h) with h = psi_up + S A psi_dn: the link multiplies
// only the projected 2-spinor h (the spin-projection trick of Sec. 3.2) and the lower two
// spins are rebuilt from U h.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace dwf {

enum { P_F64 = 0, P_F32 = 1, P_F16 = 2, P_BF16 = 3 };

template <int P> struct PT;
// LREALS: reals per link; SITE_LREALS: reals per site's eight links, padding included
template <> struct PT<P_F64> {
  using real = double; using chunk = double2; using lreal = double;
  // a site's links padded by 16 bytes to 1168 (73 x 16), so that the sites of a warp read their
  // broadcast entries from different banks
  static constexpr int NCH = 12, RPC = 2, LREALS = 18, SITE_LREALS = 8 * 18 + 2; static constexpr bool HALF = false;
};
template <> struct PT<P_F32> {
  using real = float; using chunk = float4; using lreal = float;
  // links padded to 20 reals (80 bytes) so that the nine complex entries load as five float4;
  // a site's eight links padded by 16 bytes to 656 (41 float4), so that sites adjacent in a
  // half-warp read their broadcast link entries from different bank groups
  static constexpr int NCH = 6, RPC = 4, LREALS = 20, SITE_LREALS = 8 * 20 + 4; static constexpr bool HALF = false;
};
template <> struct PT<P_F16> {
  using real = float; using chunk = uint4; using lreal = __half;
  static constexpr int NCH = 3, RPC = 8, LREALS = 12, SITE_LREALS = 8 * 12; static constexpr bool HALF = true;
};
template <> struct PT<P_BF16> {
  using real = float; using chunk = uint4; using lreal = __nv_bfloat16;
  static constexpr int NCH = 3, RPC = 8, LREALS = 12, SITE_LREALS = 8 * 12; static constexpr bool HALF = true;
};
// float4 per site of the FP32 link form the hop reads (as stored, or expanded from 16 bits)
constexpr int LINK_SITE_F4 = 41;

struct Field {
  void *v;
  float *nrm;  // 16-bit precisions only
};

// scalars of one CG solve, resident in device memory (FP64 throughout)
struct CGScalars {
  double rr;       // |r|^2 of the current inner residual
  double rr_old;   // previous |r|^2 (denominator of beta)
  double qq;       // |C^dag p|^2 = (p, C C^dag p)
  double beta;     // p = r + beta p
  double rmax2;    // max |r|^2 since the last restart
  double delta2;   // reliable-update threshold squared
  double target2;  // (tol |b|)^2
  double red;      // result slot of plain norm reductions
  double red2;
  double alpha;     // (r, r) / (p, A p), set by the reduction that finishes |C^dag p|^2
  float alpha_f;    // the same in FP32 for the FP32-arithmetic kernels
  float beta_f;     // beta in FP32
  double rr_start;  // |r|^2 at the last restart (divergence guard)
  double rr_min;    // smallest |r|^2 since the last restart (stall guard)
  int restart_flag;  // set on device when an FP64 restart is due (a RS_* reason); kernels then skip work
  int iter;          // inner iterations done
  int iter_cap;      // restart when iter reaches this
  int error;         // kernel error word (bounded wait gave up)
  int iter_min;      // iteration at which rr_min was reached
  int stall_iters;   // restart when rr_min has not improved for this many iterations
};

// reasons for an FP64 restart
enum { RS_NONE = 0, RS_DELTA = 1, RS_TARGET = 2, RS_CAP = 3, RS_DIVERGED = 4, RS_STALLED = 5 };

// ------------------------------------------------------------------ overlapped launches
//
// The kernels of an operator or a CG iteration are launched with programmatic stream
// serialization: a kernel whose predecessor's CTAs have all called pdl_trigger() or ended may
// start, set up what no kernel of the chain writes (the matrix along s, the tile's links and
// neighbour indices) and then waits in pdl_wait() until its predecessors have completed and
// their writes are visible.  The trigger stands at the end of a kernel's main work: there the
// set-up hides behind the last CTAs and the reduction's tail (FP32 CG iteration at 8^4x16: 40.8
// -> 36.2 us, at 16^3x32x16 429 -> 423 us).  At the start of the kernels it let later kernels'
// CTAs pile up on whatever SM had room (51.7 and 468 us).  Nothing a predecessor writes is
// read, and nothing at all is written, before pdl_wait(); field loads are plain (ld.global.nc
// promises data that is constant for the whole launch, which such a launch cannot).  Without
// the launch attribute both are no-ops.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ------------------------------------------------------------------ spinor access

template <int P>
__device__ __forceinline__ void load_sp(const Field f, long cb, int s, int Ns,
                                        typename PT<P>::real (&o)[24]) {
  using T = PT<P>;
  const typename T::chunk *b = (const typename T::chunk *)f.v + (size_t)cb * T::NCH * Ns + s;
  if constexpr (P == P_F64) {
#pragma unroll
    for (int k = 0; k < 12; ++k) { double2 c = b[(size_t)k * Ns]; o[2 * k] = c.x; o[2 * k + 1] = c.y; }
  } else if constexpr (P == P_F32) {
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      float4 c = b[(size_t)k * Ns];
      o[4 * k] = c.x; o[4 * k + 1] = c.y; o[4 * k + 2] = c.z; o[4 * k + 3] = c.w;
    }
  } else {
    const float nm = f.nrm[(size_t)cb * Ns + s];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      uint4 c = b[(size_t)k * Ns];
      uint32_t w[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float2 v;
        if constexpr (P == P_F16) v = __half22float2(*reinterpret_cast<__half2 *>(&w[j]));
        else v = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&w[j]));
        o[8 * k + 2 * j] = v.x * nm;
        o[8 * k + 2 * j + 1] = v.y * nm;
      }
    }
  }
}

template <int P>
__device__ __forceinline__ void store_sp(Field f, long cb, int s, int Ns,
                                         const typename PT<P>::real (&v)[24]) {
  using T = PT<P>;
  typename T::chunk *b = (typename T::chunk *)f.v + (size_t)cb * T::NCH * Ns + s;
  if constexpr (P == P_F64) {
#pragma unroll
    for (int k = 0; k < 12; ++k) b[(size_t)k * Ns] = make_double2(v[2 * k], v[2 * k + 1]);
  } else if constexpr (P == P_F32) {
#pragma unroll
    for (int k = 0; k < 6; ++k)
      b[(size_t)k * Ns] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
  } else {
    float mx = 0.f;
#pragma unroll
    for (int c = 0; c < 24; ++c) mx = fmaxf(mx, fabsf(v[c]));
    const float sc = mx > 0.f ? 1.0f / mx : 0.f;
    f.nrm[(size_t)cb * Ns + s] = mx;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      uint32_t w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float a = v[8 * k + 2 * j] * sc, bb = v[8 * k + 2 * j + 1] * sc;
        if constexpr (P == P_F16) { __half2 h = __floats2half2_rn(a, bb); w[j] = *reinterpret_cast<uint32_t *>(&h); }
        else { __nv_bfloat162 h = __floats2bfloat162_rn(a, bb); w[j] = *reinterpret_cast<uint32_t *>(&h); }
      }
      b[(size_t)k * Ns] = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// one 16-byte chunk k of (cb, s) (FP64: 2 reals, FP32: 4 reals); unnormalised precisions only
template <int P>
__device__ __forceinline__ void load_chunk(const Field f, long cb, int s, int Ns, int k,
                                           typename PT<P>::real (&o)[PT<P>::RPC]) {
  static_assert(!PT<P>::HALF, "chunk access needs an unnormalised precision");
  const typename PT<P>::chunk c = ((const typename PT<P>::chunk *)f.v)[((size_t)cb * PT<P>::NCH + k) * Ns + s];
  if constexpr (P == P_F64) { o[0] = c.x; o[1] = c.y; }
  else { o[0] = c.x; o[1] = c.y; o[2] = c.z; o[3] = c.w; }
}
template <int P>
__device__ __forceinline__ void store_chunk(Field f, long cb, int s, int Ns, int k,
                                            const typename PT<P>::real (&v)[PT<P>::RPC]) {
  static_assert(!PT<P>::HALF, "chunk access needs an unnormalised precision");
  typename PT<P>::chunk *b = (typename PT<P>::chunk *)f.v + ((size_t)cb * PT<P>::NCH + k) * Ns + s;
  if constexpr (P == P_F64) *b = make_double2(v[0], v[1]);
  else *b = make_float4(v[0], v[1], v[2], v[3]);
}

// ------------------------------------------------------------------ links

template <int P>
__device__ __forceinline__ void load_link(const typename PT<P>::lreal *L, typename PT<P>::real (&W)[18]) {
  if constexpr (!PT<P>::HALF) {
#pragma unroll
    for (int i = 0; i < 18; ++i) W[i] = L[i];
  } else {
#pragma unroll
    for (int i = 0; i < 12; ++i) {
      if constexpr (P == P_F16) W[i] = __half2float(L[i]);
      else W[i] = __bfloat162float(L[i]);
    }
    // third row = conj(row0 x row1) for an SU(3) matrix
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int b1 = (b + 1) % 3, b2 = (b + 2) % 3;
      // (r0 x r1)_b = r0_{b1} r1_{b2} - r0_{b2} r1_{b1}
      float re = (W[2 * b1] * W[6 + 2 * b2] - W[2 * b1 + 1] * W[6 + 2 * b2 + 1]) -
                 (W[2 * b2] * W[6 + 2 * b1] - W[2 * b2 + 1] * W[6 + 2 * b1 + 1]);
      float im = (W[2 * b1] * W[6 + 2 * b2 + 1] + W[2 * b1 + 1] * W[6 + 2 * b2]) -
                 (W[2 * b2] * W[6 + 2 * b1 + 1] + W[2 * b2 + 1] * W[6 + 2 * b1]);
      W[12 + 2 * b] = re;
      W[12 + 2 * b + 1] = -im;
    }
  }
}

// ------------------------------------------------------------------ spin projection

// A_mu = upper-right block of gamma_mu; each row of A and A^dag has one non-zero
// entry, phase code 0: 1, 1: i, 2: -1, 3: -i.
__host__ __device__ constexpr int a_col(int mu, int j) { return (mu == 0 || mu == 1) ? 1 - j : j; }
__host__ __device__ constexpr int a_ph(int mu, int j) {
  return mu == 0 ? 3 : mu == 1 ? (j == 0 ? 2 : 0) : mu == 2 ? (j == 0 ? 3 : 1) : 0;
}
__host__ __device__ constexpr int ad_col(int mu, int k) { return (mu == 0 || mu == 1) ? 1 - k : k; }
__host__ __device__ constexpr int ad_ph(int mu, int k) {
  return mu == 0 ? 1 : mu == 1 ? (k == 0 ? 0 : 2) : mu == 2 ? (k == 0 ? 1 : 3) : 0;
}

template <int PH, typename R>
__device__ __forceinline__ void phase(R &re, R &im) {
  if constexpr (PH == 1) { R t = re; re = -im; im = t; }
  else if constexpr (PH == 2) { re = -re; im = -im; }
  else if constexpr (PH == 3) { R t = re; re = im; im = -t; }
}

// ------------------------------------------------------------------ packed FP32 pairs
//
// Blackwell executes two FP32 operations per instruction on a 64-bit register pair
// (add/sub/mul/fma .rn.f32x2).  A complex number (re, im) is such a pair; a sum of
// complex products sum_b w_b h_b is two packed FMA chains, P = sum_b w_b (hr_b, hr_b) and
// Q = sum_b w_b (hi_b, hi_b), joined as P + (-1, 1) (Q.y, Q.x).

struct f2 {
  unsigned long long v;
};
__device__ __forceinline__ f2 pk2(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void upk2(f2 x, float &a, float &b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
// a * b + c
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ f2 swp2(f2 x) {
  float a, b;
  upk2(x, a, b);
  return pk2(b, a);
}

// up + S * phase(PH) * z with the sign S a run-time value, given as the packed pairs
// s2 = (S, S), ns2 = (-S, -S), sa = (-S, S), nsa = (S, -S)
struct SignPairs {
  f2 s2, ns2, sa, nsa;
};
__device__ __forceinline__ SignPairs sign_pairs(float S) {
  return SignPairs{pk2(S, S), pk2(-S, -S), pk2(-S, S), pk2(S, -S)};
}
template <int PH>
__device__ __forceinline__ f2 add_phase_rt(f2 up, f2 z, const SignPairs &sg) {
  if constexpr (PH == 0) return fma2(z, sg.s2, up);
  else if constexpr (PH == 2) return fma2(z, sg.ns2, up);
  else if constexpr (PH == 1) return fma2(swp2(z), sg.sa, up);   // i z = (-zi, zr)
  else return fma2(swp2(z), sg.nsa, up);                          // -i z = (zi, -zr)
}

// acc += (1 + S g_mu) W psi in FP32 pairs, with S = +-1 at run time (forward hops S = -1,
// backward S = +1, so the eight directions run the same instructions) and the link as
// stored (nine complex entries, pairs of them 16-byte aligned):
// W h = P + (-1, 1) (Q.y, Q.x) with P = sum_b W_b (hr_b, hr_b), Q = sum_b W_b (hi_b, hi_b)
template <int MU>
__device__ __forceinline__ void hop_dir_raw(f2 (&acc)[12], const f2 (&ps)[12], const float4 *Wl,
                                            const SignPairs &sg) {
  f2 hr[2][3], hi[2][3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const f2 h0 = add_phase_rt<a_ph(MU, 0)>(ps[a], ps[a + 3 * (2 + a_col(MU, 0))], sg);
    const f2 h1 = add_phase_rt<a_ph(MU, 1)>(ps[a + 3], ps[a + 3 * (2 + a_col(MU, 1))], sg);
    float x, y;
    upk2(h0, x, y);
    hr[0][a] = pk2(x, x);
    hi[0][a] = pk2(y, y);
    upk2(h1, x, y);
    hr[1][a] = pk2(x, x);
    hi[1][a] = pk2(y, y);
  }
  const f2 sgn = pk2(-1.f, 1.f);
  float4 w1;  // row 0 ends and row 1 starts in the second float4
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    f2 W0, W1, W2;  // row a: entries 3a, 3a + 1, 3a + 2
    if (a == 0) {
      const float4 w0 = Wl[0];
      w1 = Wl[1];
      W0 = pk2(w0.x, w0.y), W1 = pk2(w0.z, w0.w), W2 = pk2(w1.x, w1.y);
    } else if (a == 1) {
      const float4 w2 = Wl[2];
      W0 = pk2(w1.z, w1.w), W1 = pk2(w2.x, w2.y), W2 = pk2(w2.z, w2.w);
    } else {
      const float4 w3 = Wl[3], w4 = Wl[4];
      W0 = pk2(w3.x, w3.y), W1 = pk2(w3.z, w3.w), W2 = pk2(w4.x, w4.y);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      f2 P = mul2(W0, hr[j][0]);
      P = fma2(W1, hr[j][1], P);
      P = fma2(W2, hr[j][2], P);
      f2 Q = mul2(W0, hi[j][0]);
      Q = fma2(W1, hi[j][1], Q);
      Q = fma2(W2, hi[j][2], Q);
      const f2 wh = fma2(sgn, swp2(Q), P);
      acc[a + 3 * j] = add2(acc[a + 3 * j], wh);
      if (ad_col(MU, 0) == j) acc[a + 6] = add_phase_rt<ad_ph(MU, 0)>(acc[a + 6], wh, sg);
      if (ad_col(MU, 1) == j) acc[a + 9] = add_phase_rt<ad_ph(MU, 1)>(acc[a + 9], wh, sg);
    }
  }
}

// ------------------------------------------------------------------ FP64 hop in fixed point
//
// GB300 issues two FP64 operations per clock and SM but sixty 32 x 32 + 64 bit integer
// multiply-adds (measured: DFMA 1.99, DADD 1.67, IMAD.WIDE 60 per clock and SM), so the
// FP64 hop forms its SU(3) products in integers.  Per (site, s) the projected half-spinors h
// are formed in FP64 as before (Eq. 12), then brought to the exponent E = the largest among
// the neighbours so far (plus one bit, so that E seldom has to grow): h = V 2^(E - 1080),
// |V| < 2^58.  Links are in units of 2^-60.  Both are split into 30-bit halves that carry the
// sign, V = hi 2^30 + lo, and a product sum over the six real terms of a row is
//   sum W V / 2^60 = sum Wh Vh + (sum (Wh Vl + Wl Vh)) / 2^30,
// three 64-bit multiply-adds per real product; the dropped Wl Vl are below one unit each.
// Bounds: a link row's 2-norm is at most sqrt(1.01) (checked; SU(3) rows have norm 1), so a
// row's result is below sqrt(1.01 * 6) 2^58 < 2^59.4 and the sum over eight directions below
// 2^62.4; the cross terms are below 6 (2^60 + 2^58) < 2^63.  The error is about one unit per
// direction, 2^-56 of the largest |h| of the (site, s): half of FP64's own rounding of the
// same sums by norm, on Gaussian fields; single components that are far smaller are looked
// after below (FX_SEEN).  Links or neighbours outside the bounds (not finite, or exponents
// outside [FX_EMIN, FX_EMAX]) take the FP64 arithmetic (hop_site_f64).  Which arithmetic a (site,
// s) takes, and its result, follow from its own links and neighbours alone: not from the order
// of the sites or the tile it is in, nor from whether a neighbour is stored as a spinor or, in
// a halo slot, as its projection.

constexpr int FX_EMIN = 80, FX_EMAX = 2000;

// The unit follows the largest |h| among all twelve reals and eight neighbours, so a colour and
// spin far below that one would keep few digits where the links do not mix it with the large ones
// (unit or diagonal links).  A complex component of the result is therefore `seen` (a bit of
// FX_SEEN each, colour + 3 spin) once a backward hop adds at least 2^53 units to it, against an
// error of one unit a hop (root mean square; ten at most): no more than FP64 makes of the same
// terms.  (E grows by two bits at least; the first such growth keeps what was seen, a second or
// a larger one does not.)  Components that are not seen then count as such if they are 2^53 in
// the result, or if fixed_loses finds that their terms' sizes are or that they have no term;
// else the (site, s) takes plain FP64.  Testing the four backward hops finds all components of
// Gaussian fields on SU(3) links but for one (site, s) in 40,000 (D^EO on 16^4 x 16
// 352 -> 359 us; a field that falls by e a slice 353 -> 450).  2^54 would send one warp in eight of a
// Gaussian field to fixed_loses (436 us), without a smaller root-mean-square error.
constexpr unsigned FX_SEEN = 0xfff, FX_GREW = 0x1000, FX_BAD = 0x2000;
constexpr int FX_SEEN_HI = 1 << 21;  // 2^53 in the upper word
// int4 per site of the fixed-point links: 8 links x 9 entries {re hi, re lo, im hi, im lo}, in the
// place of the links as copied; the site's padding, 0 as stored, is set where a row is out of bounds
constexpr int FX_SITE_I4 = PT<P_F64>::SITE_LREALS / 2;

// V = x 2^(1075 + L - E), truncated, as V = hi 2^30 + lo; E is at least x's exponent field (an x
// above it gives 0, and so do FP64 zeros and denormals)
template <int L>
__device__ __forceinline__ void to_fixed(double x, int E, int &hi, int &lo) {
  const int xh = __double2hiint(x);
  const unsigned mh = (xh & 0xfffff) | 0x100000;
  const unsigned sh = min((unsigned)(E - ((xh >> 20) & 0x7ff)), 63u);
  const unsigned long long m = ((unsigned long long)mh << 32 | (unsigned)__double2loint(x)) << L >> sh;
  const int sg = (xh >> 31) | 1;
  hi = (int)(m >> 30) * sg;
  lo = (int)(m & 0x3fffffffu) * sg;
}

// c + a b, the full 64-bit product
__device__ __forceinline__ long long mad_w(int a, int b, long long c) { return (long long)a * b + c; }

// either real is 2^53 units or more
__device__ __forceinline__ bool fx_big(long long re, long long im) {
  return (((unsigned)(int)(re >> 32) + FX_SEEN_HI) | ((unsigned)(int)(im >> 32) + FX_SEEN_HI)) >= 2u * FX_SEEN_HI;
}

// h_j = psi_up + S A psi_dn of direction MU (spin projection), FP64; one multiply-add a real (the
// FP64 pipe issues DFMA faster than DADD, and a product with +-1 is exact)
template <int MU>
__device__ __forceinline__ void project_f64(const double (&ps)[24], double S, double (&h)[12]) {
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const int src = 2 * (a + 3 * (2 + a_col(MU, j))), dst = 2 * (a + 3 * j);
      // phase code 0: 1, 1: i, 2: -1, 3: -i
      const int p = a_ph(MU, j);
      const double vr = (p & 1) ? ps[src + 1] : ps[src], vi = (p & 1) ? ps[src] : ps[src + 1];
      h[dst] = fma((p == 1 || p == 2) ? -S : S, vr, ps[dst]);
      h[dst + 1] = fma((p == 2 || p == 3) ? -S : S, vi, ps[dst + 1]);
    }
}

// acc += (1 + S g_MU) W psi in units of 2^(E - 1080); W: the link's nine entries; st: FX_SEEN,
// FX_GREW, FX_BAD (a value is outside the fixed-point range, acc is then meaningless)
template <int MU>
__device__ __forceinline__ void hop_dir_fixed(long long (&acc)[24], int &E, unsigned &st, const double (&ps)[24],
                                              const int4 *W, const bool back) {
  double h[12];
  project_f64<MU>(ps, back ? 1.0 : -1.0, h);
  int em = 0;
#pragma unroll
  for (int q = 0; q < 12; ++q) em = max(em, __double2hiint(h[q]) & 0x7fffffff);
  em >>= 20;
  if (em > FX_EMAX) st |= FX_BAD;
  if (__builtin_expect(em < FX_EMIN, 0)) {  // all zero (nothing to add), or too small for the fixed-point range
    unsigned any = 0;
#pragma unroll
    for (int q = 0; q < 12; ++q) any |= (unsigned)(__double2hiint(h[q]) << 1) | (unsigned)__double2loint(h[q]);
    if (any) st |= FX_BAD;
  }
  if (__builtin_expect(em > E, 0)) {
    const int d = min(em + 1 - E, 63);
#pragma unroll
    for (int c = 0; c < 24; ++c) acc[c] >>= d;
    E = em + 1;
    if (d == 2 && !(st & FX_GREW)) st |= FX_GREW;
    else st &= FX_BAD;
  }
  int ph[6], pl[6], qh[6], ql[6], nh[6], nl[6];  // real parts, imaginary parts, - imaginary parts
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    to_fixed<5>(h[2 * q], E, ph[q], pl[q]);
    to_fixed<5>(h[2 * q + 1], E, qh[q], ql[q]);
    nh[q] = -qh[q];
    nl[q] = -ql[q];
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int4 w[3] = {W[3 * a], W[3 * a + 1], W[3 * a + 2]};
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      long long Hr = 0, Hi = 0, Xr = 1 << 29, Xi = 1 << 29;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const int q = 3 * j + b;
        Hr = mad_w(w[b].z, nh[q], mad_w(w[b].x, ph[q], Hr));
        Hi = mad_w(w[b].z, ph[q], mad_w(w[b].x, qh[q], Hi));
        Xr = mad_w(w[b].w, nh[q], mad_w(w[b].z, nl[q], mad_w(w[b].y, ph[q], mad_w(w[b].x, pl[q], Xr))));
        Xi = mad_w(w[b].w, ph[q], mad_w(w[b].z, pl[q], mad_w(w[b].y, qh[q], mad_w(w[b].x, ql[q], Xi))));
      }
      const long long re = Hr + (Xr >> 30), im = Hi + (Xi >> 30);
      const int u = 2 * (a + 3 * j);
      acc[u] += re;
      acc[u + 1] += im;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (ad_col(MU, k) != j) continue;
        if (back && fx_big(re, im)) st |= 1u << (a + 3 * j) | 1u << (a + 3 * (2 + k));
        const int dn = 2 * (a + 3 * (2 + k)), p = ad_ph(MU, k);
        // S phase (re + i im): phase 0: 1, 1: i, 2: -1, 3: -i
        const long long vr = (p & 1) ? im : re, vi = (p & 1) ? re : im;
        acc[dn] = (p == 1 || p == 2) == back ? acc[dn] - vr : acc[dn] + vr;
        acc[dn + 1] = (p == 2 || p == 3) == back ? acc[dn + 1] - vi : acc[dn + 1] + vi;
      }
    }
  }
}

// a 2^(k - 1023), rounded to nearest even: as (double)a times a power of two, without the two
// instructions on the FP64 pipe (C C^dag in FP64 at 16^3x32x16: 2.98 -> 2.83 ms)
__device__ __forceinline__ double from_fixed(long long a, int k) {
  const unsigned long long u = a < 0 ? -(unsigned long long)a : (unsigned long long)a;
  const int z = __clzll((long long)u);
  const unsigned long long n = u << (z & 63);  // leading one at bit 63
  // 53 bits with their exponent, and the rest rounded (a carry moves into the exponent)
  unsigned long long r = (n >> 11) + ((unsigned long long)(k + 62 - z) << 52);
  const unsigned rest = (unsigned)n & 0x7ffu;
  r += (rest + 0x3ffu + (unsigned)(r & 1)) >> 11;
  r |= (unsigned long long)a & 0x8000000000000000ull;
  return u ? __longlong_as_double((long long)r) : 0.0;
}

// a link row (three complex entries) to units of 2^-60, split as above, in place: an entry {re hi,
// re lo, im hi, im lo} takes its two doubles' 16 bytes; false if its 2-norm is out of bounds or
// not a number
__device__ __forceinline__ bool link_row_fixed(double2 *w) {
  float n2 = 0.f;
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    const double2 u = w[b];
    n2 += (float)u.x * (float)u.x + (float)u.y * (float)u.y;
    int xh, xl, yh, yl;
    to_fixed<8>(u.x, 1023, xh, xl);
    to_fixed<8>(u.y, 1023, yh, yl);
    w[b] = make_double2(__hiloint2double(xl, xh), __hiloint2double(yl, yh));
  }
  return n2 <= 1.01f;
}

// the same in plain FP64 with the sign S at run time, for values out of the fixed-point range
template <int MU, typename R>
__device__ __forceinline__ void hop_dir_s(R (&acc)[24], const R (&ps)[24], const R (&W)[18], R S) {
  R h[2][3][2];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int src = 2 + a_col(MU, j);
      R vr = ps[2 * (a + 3 * src)], vi = ps[2 * (a + 3 * src) + 1];
      switch (a_ph(MU, j)) {
        case 1: { R t = vr; vr = -vi; vi = t; } break;
        case 2: vr = -vr; vi = -vi; break;
        case 3: { R t = vr; vr = vi; vi = -t; } break;
        default: break;
      }
      h[j][a][0] = ps[2 * (a + 3 * j)] + S * vr;
      h[j][a][1] = ps[2 * (a + 3 * j) + 1] + S * vi;
    }
  }
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      R re = 0, im = 0;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const R ur = W[2 * (3 * a + b)], ui = W[2 * (3 * a + b) + 1];
        re += ur * h[j][b][0] - ui * h[j][b][1];
        im += ur * h[j][b][1] + ui * h[j][b][0];
      }
      acc[2 * (a + 3 * j)] += re;
      acc[2 * (a + 3 * j) + 1] += im;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        if (ad_col(MU, k) != j) continue;
        R vr = re, vi = im;
        switch (ad_ph(MU, k)) {
          case 1: { R t = vr; vr = -vi; vi = t; } break;
          case 2: vr = -vr; vi = -vi; break;
          case 3: { R t = vr; vr = vi; vi = -t; } break;
          default: break;
        }
        acc[2 * (a + 3 * (2 + k))] += S * vr;
        acc[2 * (a + 3 * (2 + k)) + 1] += S * vi;
      }
    }
}

}  // namespace dwf
