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
// Ns - 1 - j for a chirality that runs backward), three FP64 operations a real and step and one
// for the closure, against Ns for the dense row:
//   u_j = A_j v_j + y_j,  y_{j+1} = D_j v_j - E_j y_j,  y_0 = sum_j W_j v_j (the closure, through
// the corner kappa of L, Eq. 4).  The diagonal term enters u last, so u takes one rounding and
// those of the smaller y
enum { RC_A, RC_D, RC_E, RC_W, RC_N = 4 };

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

// a number as the sum of two doubles, for the table entries: each then is within half a unit of
// its last place, where products and quotients of rounded factors lose two or three units
struct Dd {
  double h, l;
  Dd(double x = 0.0) : h(x), l(0.0) {}
  Dd(double x, double y) : h(x + y), l(y - ((x + y) - x)) {}  // |x| >= |y|
};
inline Dd operator-(const Dd &a) {
  Dd r;
  r.h = -a.h, r.l = -a.l;
  return r;
}
inline Dd operator+(const Dd &a, const Dd &b) {
  const double s = a.h + b.h, t = s - a.h;
  return Dd(s, ((a.h - (s - t)) + (b.h - t)) + (a.l + b.l));
}
inline Dd operator-(const Dd &a, const Dd &b) { return a + -b; }
inline Dd operator*(const Dd &a, const Dd &b) {
  const double p = a.h * b.h;
  return Dd(p, std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
inline Dd operator/(const Dd &a, const Dd &b) {
  const double q = a.h / b.h;
  return Dd(q, (a - b * Dd(q)).h / b.h);
}
inline Dd sqrt_dd(double x) {
  const double r = std::sqrt(x);
  return Dd(r, std::fma(-r, r, x) / (2.0 * r));
}

// u = the recurrence of table T (one chirality) applied to v, operation for operation as the kernels
inline void apply_recurrence(const double *T, int Ns, bool bwd, const double *v, double *u) {
  auto sg = [&](int j) { return bwd ? Ns - 1 - j : j; };
  double y = 0.0;
  for (int j = 0; j < Ns; ++j) y = std::fma(T[j * RC_N + RC_W], v[sg(j)], y);
  for (int j = 0; j < Ns; ++j) {
    const double *t = T + j * RC_N;
    const double x = v[sg(j)];
    u[sg(j)] = std::fma(t[RC_A], x, y);
    y = std::fma(-t[RC_E], y, t[RC_D] * x);
  }
}

// one chirality's table.  With den = (d - m0) omega + 1, g = (sigma + omega) / (omega den) and
// n, k the slices of the step before and after this one (at s):
//   M5 = P A^{-1} (Eq. 8, P = sqrt(omega) (1 + cL)): A z = v in steps z = A_j v - C_j z', C =
//     ((d - m0) sigma - 1) / den sqrt(omega / omega_n), then u = A_j v + G_j z' with G = g
//     sqrt(omega / omega_n); y = G_j z' is kept, so that A = omega / den, D = G_{j+1} A_j, E =
//     C_j G_{j+1} / G_j.  A step whose G is 0 or negligible (sigma = - omega) keeps 2^-60 of
//     what it would be with |sigma| instead, which is below u's rounding.  S1 = M5 omega^{-1/2} scales A and D.
//   M5^T = A^{-T} P^T: A as above, D = g sqrt(omega omega_k) / den_k, E = ((d - m0) sigma - 1) /
//     den_k sqrt(omega_k / omega)
//   S2 = (1 + cL)^{-1} omega^{-1/2} (Eq. 9): A = omega^{-1/2}, E = c_k = sigma_k / omega_k, D = - E A
//   the bidiagonal matrices of Eq. 5: A the diagonal, D the factor of L at k, E = 0
// false if the closure has no solution.
inline bool recurrence_table(const SMatrices &c, int kind, int chi, double *T) {
  const int Ns = c.Ns;
  const bool bwd = (chi ^ (kind == MK_M5T)) != 0;
  auto sg = [&](int j) { return bwd ? Ns - 1 - j : j; };
  const Dd kappa = -(Dd(c.mq) / Dd(2.0 * c.m0)), dm = Dd(kD) - Dd(c.m0);
  std::vector<Dd> A(Ns), D(Ns), E(Ns), G(Ns);
  auto om = [&](int j) { return Dd(c.omega[sg(j)]); };
  auto si = [&](int j) { return Dd(c.sigma[sg(j)]); };
  auto rt = [&](int j) { return sqrt_dd(c.omega[sg(j)]); };
  auto den = [&](int j) { return dm * om(j) + Dd(1.0); };
  auto g = [&](int j) { return (si(j) + om(j)) / (om(j) * den(j)); };
  for (int j = 0; j < Ns; ++j) {
    const Dd x = rt(j) / rt((j + Ns - 1) % Ns);
    const double least = std::ldexp((std::fabs(si(j).h) + om(j).h) / (om(j) * den(j) * x).h, -60);
    G[j] = g(j) * x;
    if (!(std::fabs(G[j].h) > least)) G[j] = Dd(least);
  }
  for (int j = 0; j < Ns; ++j) {
    const int k = (j + 1) % Ns, n = (j + Ns - 1) % Ns;
    switch (kind) {
      case MK_M5:
      case MK_S1:
        A[j] = (kind == MK_M5 ? om(j) : rt(j)) / den(j);
        D[j] = G[k] * A[j];
        E[j] = (dm * si(j) - Dd(1.0)) / den(j) * (rt(j) / rt(n)) * (G[k] / G[j]);
        break;
      case MK_M5T:
        A[j] = om(j) / den(j);
        D[j] = g(j) * rt(j) * rt(k) / den(k);
        E[j] = (dm * si(j) - Dd(1.0)) / den(k) * (rt(k) / rt(j));
        break;
      case MK_S2:
        A[j] = Dd(1.0) / rt(j);
        E[j] = si(k) / om(k);
        D[j] = -(E[j] * A[j]);
        break;
      case MK_W: A[j] = om(j), D[j] = si(k); break;                                            // omega + sigma L
      case MK_Z: A[j] = dm * om(j) + Dd(1.0), D[j] = dm * si(k) - Dd(1.0); break;  // (d - m0) of it + 1 - L
      case MK_ID: A[j] = Dd(1.0); break;
      case MK_MASS: A[j] = dm; break;
    }
  }
  // closure: y_0 = kappa y_Ns, where y_Ns depends linearly on y_0 through every step
  Dd q = kappa;
  for (int j = 0; j < Ns; ++j) q = q * -E[j];
  const Dd one_q = Dd(1.0) - q;
  if (one_q.h == 0.0) return false;
  Dd r = kappa / one_q;
  for (int j = Ns - 1; j >= 0; --j) {
    const Dd w = r * D[j];
    r = r * -E[j];
    if (Ns == 1) A[j] = A[j] + w;  // a single slice: one product
    T[j * RC_N + RC_A] = A[j].h;
    T[j * RC_N + RC_D] = Ns == 1 ? 0.0 : D[j].h;
    T[j * RC_N + RC_E] = Ns == 1 ? 0.0 : E[j].h;
    T[j * RC_N + RC_W] = Ns == 1 ? 0.0 : w.h;
  }
  return true;
}

// builds the tables and checks those with a solve against their dense matrices column by
// column; S1 and S2 may have none, M5 and M5^T have to agree.  The bidiagonal matrices are
// their tables' own entries, exact for every mass and weight, and always have one: the corner
// of the dense Z, dm (sigma kappa) - kappa, cancels where dm sigma is near 1 and kappa large,
// and says nothing about the table's (dm sigma - 1) kappa.
//
// A table is tight, and the s-mixing kernel takes it, if it agrees with the dense matrix to the
// latter's own few roundings and y_0's rounding, carried along s by the product of the E, stays
// below the largest entry's.  Where sigma > omega that product grows along s and the dense rows
// are the more accurate.  Tight tables err less than the rows (root mean square over random
// fields, in units of 2^-52 of the result, M5, M5^T and S1 at Ns = 4 to 64: Shamir 0.24 against
// 0.5-0.9, Borici 0.27-0.29 against 0.4-1.0, cosine 0.30-0.37 against 0.6-1.1).
inline bool build_recurrences(SMatrices *c) {
  const int Ns = c->Ns;
  std::vector<double> u(Ns), v(Ns);
  for (int kind = 0; kind < MK_COUNT; ++kind) {
    std::vector<double> &rec = c->rec[kind];
    rec.assign((size_t)2 * Ns * RC_N, 0.0);
    bool ok = true, tight = true;
    double worst = 0.0;
    for (int chi = 0; chi < 2 && ok; ++chi) {
      double *T = rec.data() + (size_t)chi * Ns * RC_N;
      ok = recurrence_table(*c, kind, chi, T);
      if (!ok || kind >= MK_W) continue;
      const double *M = c->mat[kind].data() + (size_t)chi * Ns * Ns;
      double mmax = 0.0, wsum = 0.0, grow = 1.0, prod = 1.0;
      for (int i = 0; i < Ns * Ns; ++i) mmax = std::max(mmax, fabs(M[i]));
      for (int j = 0; j < Ns; ++j) {
        wsum += fabs(T[j * RC_N + RC_W]);
        grow = std::max(grow, prod);
        prod *= fabs(T[j * RC_N + RC_E]);
      }
      tight = tight && (grow <= 1.0 || wsum * grow <= mmax);
      for (int t0 = 0; t0 < Ns; ++t0) {
        std::fill(v.begin(), v.end(), 0.0);
        v[t0] = 1.0;
        apply_recurrence(T, Ns, (chi ^ (kind == MK_M5T)) != 0, v.data(), u.data());
        for (int s = 0; s < Ns; ++s)
          worst = std::max(worst, std::isfinite(u[s]) ? fabs(u[s] - M[s * Ns + t0]) / mmax : 1.0);
      }
    }
    // (a system is refused where the two differ by more: too ill conditioned for either)
    if (!ok || worst > 2e-11) {
      if (kind == MK_M5 || kind == MK_M5T) return false;
      rec.clear();
    }
    c->rec_tight[kind] = ok && tight && worst <= 1e-15;
  }
  return true;
}

}  // namespace dwf
