// dwf_smat.h -- the matrices along the fifth dimension of one system (host code, no CUDA
// types): dense, and as the recurrence tables of the FP64 kernels.  They follow from Ns, the
// masses and the weights alone, so they can be built and tested without a GPU.
#pragma once

#include <algorithm>
#include <cmath>
#include <vector>

namespace dwf {

constexpr double kD = 4.0;  // space-time dimension d of Eq. 2

// matrices along s held per context (kernel order K[chi][t][s] on the device); those from MK_W
// on are cyclic bidiagonal
enum MatKind { MK_M5 = 0, MK_M5T, MK_S1, MK_S2, MK_W, MK_Z, MK_ID, MK_MASS, MK_COUNT };

// FP64 recurrence along s (one table per matrix: per chirality Ns steps, step j at s = j, or
// Ns - 1 - j for a chirality that runs backward), two or three FP64 operations a real and step
// and one for the closure, against Ns for the dense row:
//   z_j = A_j v_j + B_j v_{j-1} - C_j z_{j-1},  u_j = z_j + R_j z_{j-1},
// where step 0 takes v_{-1} = kappa v_{Ns-1} and z_{-1} = kappa z_{Ns-1}, with z_{Ns-1} known
// beforehand from the closure z_{Ns-1} = sum_j W_j v_j
enum { RC_A, RC_B, RC_C, RC_R, RC_W, RC_N = 6 };

struct SMatrices {
  int Ns = 0;
  double m0 = 0, mq = 0;
  std::vector<double> omega, sigma;
  // host FP64 matrices, row-major [chi][s][t]
  std::vector<double> mat[MK_COUNT];
  // the same as FP64 recurrence tables along s (RC_A); empty where there is none
  std::vector<double> rec[MK_COUNT];
  bool rec_tight[MK_COUNT] = {};  // as accurate as the dense matrix: used by s-mixing too
};

// M5 of Eq. 8 is applied as a dense Ns x Ns matrix per chirality (Sec. 3.3).  Its entries
// are computed here column by column from the structure of Eq. 8: with y = omega^{-1/2} u
// and z = (1 + cL)^{-1} y, M5^{-1} u = v becomes the cyclic bidiagonal system
//   [(d - m0) sqrt(omega) + 1/sqrt(omega)] z + [(d - m0) sigma/sqrt(omega) - 1/sqrt(omega)] L z = v,
// then u = sqrt(omega) (z + c L z).  L = L+ (chirality +) or L- (chirality -), Eq. 4.

// (A + B L) z = v for the cyclic shift L of Eq. 4: chirality 0 uses L+ ((L z)_s = z_{s-1},
// (L z)_0 = kappa z_{Ns-1}), chirality 1 uses L- = L+^T.  Returns false on a zero pivot.
inline bool cyclic_solve(int Ns, const double *A, const double *B, double kappa, int chi, const double *v,
                         double *z) {
  std::vector<double> al(Ns), be(Ns);
  auto at = [&](int k) { return chi == 0 ? k : Ns - 1 - k; };
  const int s0 = at(0), last = at(Ns - 1);
  al[s0] = 0.0;
  be[s0] = 1.0;
  for (int k = 1; k < Ns; ++k) {
    const int s = at(k), sp = at(k - 1);
    if (A[s] == 0.0) return false;
    al[s] = (v[s] - B[s] * al[sp]) / A[s];
    be[s] = -B[s] * be[sp] / A[s];
  }
  const double den = A[s0] + B[s0] * kappa * be[last];
  if (den == 0.0) return false;
  const double zeta = (v[s0] - B[s0] * kappa * al[last]) / den;
  for (int s = 0; s < Ns; ++s) z[s] = al[s] + be[s] * zeta;
  return true;
}

// (L z)_s for chirality chi
inline double lshift(int Ns, double kappa, int chi, const double *z, int s) {
  if (chi == 0) return s > 0 ? z[s - 1] : kappa * z[Ns - 1];
  return s < Ns - 1 ? z[s + 1] : kappa * z[0];
}

inline bool build_matrices(SMatrices *c) {
  const int Ns = c->Ns;
  const double kappa = -c->mq / (2.0 * c->m0);
  const double dm = kD - c->m0;
  for (auto &m : c->mat) m.assign((size_t)2 * Ns * Ns, 0.0);
  std::vector<double> A(Ns), B(Ns), A1(Ns), Bc(Ns), v(Ns), z(Ns);
  for (int s = 0; s < Ns; ++s) {
    const double rw = sqrt(c->omega[s]);
    A[s] = dm * rw + 1.0 / rw;
    B[s] = dm * c->sigma[s] / rw - 1.0 / rw;
    A1[s] = 1.0;
    Bc[s] = c->sigma[s] / c->omega[s];
  }
  for (int chi = 0; chi < 2; ++chi) {
    double *M5 = c->mat[MK_M5].data() + (size_t)chi * Ns * Ns;
    double *M5T = c->mat[MK_M5T].data() + (size_t)chi * Ns * Ns;
    double *S1 = c->mat[MK_S1].data() + (size_t)chi * Ns * Ns;
    double *S2 = c->mat[MK_S2].data() + (size_t)chi * Ns * Ns;
    double *W = c->mat[MK_W].data() + (size_t)chi * Ns * Ns;
    double *Z = c->mat[MK_Z].data() + (size_t)chi * Ns * Ns;
    double *ID = c->mat[MK_ID].data() + (size_t)chi * Ns * Ns;
    double *MS = c->mat[MK_MASS].data() + (size_t)chi * Ns * Ns;
    for (int j = 0; j < Ns; ++j) {
      std::fill(v.begin(), v.end(), 0.0);
      v[j] = 1.0;
      // column j of M5
      if (!cyclic_solve(Ns, A.data(), B.data(), kappa, chi, v.data(), z.data())) return false;
      for (int s = 0; s < Ns; ++s)
        M5[s * Ns + j] = sqrt(c->omega[s]) * (z[s] + Bc[s] * lshift(Ns, kappa, chi, z.data(), s));
      // column j of (1 + cL)^{-1}, for S2 = Y^{-1} sqrt(omega) = (1 + cL)^{-1} omega^{-1/2} (Eq. 9)
      if (!cyclic_solve(Ns, A1.data(), Bc.data(), kappa, chi, v.data(), z.data())) return false;
      for (int s = 0; s < Ns; ++s) S2[s * Ns + j] = z[s] / sqrt(c->omega[j]);
    }
    for (int s = 0; s < Ns; ++s)
      for (int t = 0; t < Ns; ++t) {
        M5T[s * Ns + t] = M5[t * Ns + s];
        S1[s * Ns + t] = M5[s * Ns + t] / sqrt(c->omega[t]);  // S1 = M5 omega^{-1/2}
        // L_{st} of Eq. 4 for this chirality
        double Lst;
        if (chi == 0) Lst = (s > 0 ? (t == s - 1) : (t == Ns - 1) * kappa);
        else Lst = (s < Ns - 1 ? (t == s + 1) : (t == 0) * kappa);
        if (Ns == 1) Lst = kappa;
        const double diag = (s == t) ? 1.0 : 0.0;
        W[s * Ns + t] = c->omega[s] * diag + c->sigma[s] * Lst;  // omega + sigma L
        Z[s * Ns + t] = dm * W[s * Ns + t] + diag - Lst;          // (d - m0) W + 1 - L
        ID[s * Ns + t] = diag;
        MS[s * Ns + t] = dm * diag;
      }
  }
  for (auto &m : c->mat)
    for (double x : m)
      if (!std::isfinite(x)) return false;
  return true;
}

// The fifth-dimension matrices as recurrences along s for the FP64 kernels (tables of RC_A).
// With A = (d - m0) sqrt(omega) (1 + cL) + omega^{-1/2} (1 - L) (cyclic bidiagonal through the
// corner kappa of L, Eq. 4; diagonal a, below it beta) and P = sqrt(omega) (1 + cL):
// M5 = P A^{-1}, M5^T = A^{-T} P^T (Eq. 8), S1 = M5 omega^{-1/2}, S2 = (1 + cL)^{-1}
// omega^{-1/2} (Eq. 9); and the bidiagonal matrices of Eq. 5.  A chirality's recurrence visits
// s in one direction (step j at s = j, or Ns - 1 - j when backward: chirality - , or chirality
// + for M5^T).  In P A^{-1} the solved z is kept as sqrt(omega) z, which leaves one
// multiplication per step for P.
inline void apply_recurrence(const double *T, int Ns, bool bwd, double kappa, const double *v, double *u) {
  auto sg = [&](int j) { return bwd ? Ns - 1 - j : j; };
  double zc = 0.0;
  for (int j = 0; j < Ns; ++j) zc += T[j * RC_N + RC_W] * v[sg(j)];
  double zp = kappa * zc, vp = kappa * v[sg(Ns - 1)];
  for (int j = 0; j < Ns; ++j) {
    const double *t = T + j * RC_N;
    const int s = sg(j);
    const double z = t[RC_A] * v[s] + t[RC_B] * vp - t[RC_C] * zp;
    u[s] = z + t[RC_R] * zp;
    zp = z;
    vp = v[s];
  }
}

// builds the tables and checks those with a solve against their dense matrices column by
// column; S1 and S2 may have none, M5 and M5^T have to agree.  The bidiagonal matrices are
// their tables' own entries, exact for every mass and weight, and always have one: the corner
// of the dense Z, dm (sigma kappa) - kappa, cancels where dm sigma is near 1 and kappa large,
// and says nothing about the table's (dm sigma - 1) kappa
inline bool build_recurrences(SMatrices *c) {
  const int Ns = c->Ns;
  const double kappa = -c->mq / (2.0 * c->m0);
  const double dm = kD - c->m0;
  std::vector<double> a(Ns), beta(Ns), sw(Ns), cc(Ns), lam(Ns), u(Ns), v(Ns);
  for (int s = 0; s < Ns; ++s) {
    sw[s] = sqrt(c->omega[s]);
    a[s] = dm * sw[s] + 1.0 / sw[s];
    beta[s] = dm * c->sigma[s] / sw[s] - 1.0 / sw[s];
    cc[s] = c->sigma[s] / c->omega[s];
    if (a[s] == 0.0) return false;
  }
  for (int kind = 0; kind < MK_COUNT; ++kind) {
    std::vector<double> &rec = c->rec[kind];
    rec.assign((size_t)2 * Ns * RC_N, 0.0);
    double worst = 0.0;
    bool ok = true;
    for (int chi = 0; chi < 2 && ok; ++chi) {
      const bool bwd = (chi ^ (kind == MK_M5T)) != 0;
      auto sg = [&](int j) { return bwd ? Ns - 1 - j : j; };
      double *T = rec.data() + (size_t)chi * Ns * RC_N;
      for (int j = 0; j < Ns; ++j) {
        const int s = sg(j), n = sg((j + Ns - 1) % Ns);  // this step's s and the step before's
        double *t = T + j * RC_N;
        if (kind == MK_M5T) {  // g = P^T v, then A^T z = g
          t[RC_A] = sw[s] / a[s];
          t[RC_B] = sw[n] * cc[n] / a[s];
          t[RC_C] = beta[n] / a[s];
        } else if (kind == MK_W || kind == MK_Z) {  // omega + sigma L; (d - m0) of it + 1 - L
          t[RC_A] = kind == MK_W ? c->omega[s] : dm * c->omega[s] + 1.0;
          t[RC_B] = kind == MK_W ? c->sigma[s] : dm * c->sigma[s] - 1.0;
        } else if (kind == MK_ID || kind == MK_MASS) {
          t[RC_A] = kind == MK_ID ? 1.0 : dm;
        } else if (kind == MK_S2) {  // (1 + cL) z = omega^{-1/2} v
          t[RC_A] = 1.0 / sw[s];
          t[RC_C] = cc[s];
        } else {  // A z = v (S1: omega^{-1/2} v), u = sqrt(omega) (z + c L z); sqrt(omega) z kept
          t[RC_A] = (kind == MK_S1 ? 1.0 : sw[s]) / a[s];
          t[RC_C] = beta[s] / a[s] * sw[s] / sw[n];
          t[RC_R] = cc[s] * sw[s] / sw[n];
        }
      }
      // closure: z_last depends linearly on z_{-1} = kappa z_last through every step
      double q = -T[RC_C] * kappa;
      for (int j = 1; j < Ns; ++j) q *= -T[j * RC_N + RC_C];
      const double den = 1.0 - q;
      ok = den != 0.0;
      double r = 1.0;
      for (int j = Ns - 1; j >= 0 && ok; --j) {
        lam[j] = r / den;
        r *= -T[j * RC_N + RC_C];
      }
      for (int j = 0; j < Ns && ok; ++j) {
        double w = lam[j] * T[j * RC_N + RC_A];
        if (j + 1 < Ns) w += lam[j + 1] * T[(j + 1) * RC_N + RC_B];
        if (j == Ns - 1) w += kappa * lam[0] * T[RC_B];
        T[j * RC_N + RC_W] = w;
      }
      // check: the recurrence reproduces every column of the dense matrix
      const double *M = c->mat[kind].data() + (size_t)chi * Ns * Ns;
      double mmax = 0.0;
      for (int i = 0; i < Ns * Ns; ++i) mmax = std::max(mmax, fabs(M[i]));
      for (int t0 = 0; t0 < Ns && ok; ++t0) {
        std::fill(v.begin(), v.end(), 0.0);
        v[t0] = 1.0;
        apply_recurrence(T, Ns, bwd, kappa, v.data(), u.data());
        for (int s = 0; s < Ns; ++s)
          worst = std::max(worst, std::isfinite(u[s]) ? fabs(u[s] - M[s * Ns + t0]) / mmax : 1.0);
      }
    }
    if (kind >= MK_W) worst = 0.0;
    if (!ok || worst > 1e-11) {
      if (kind == MK_M5 || kind == MK_M5T) return false;
      rec.clear();
    }
    // where the recurrence grows along s (sigma > omega) it loses digits that the dense rows
    // keep: the s-mixing kernel then takes those (Shamir, Borici and cosine weights up to
    // Ns = 64 agree to 1e-15)
    c->rec_tight[kind] = ok && worst <= 1e-14;
  }
  return true;
}

}  // namespace dwf
