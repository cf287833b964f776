"""The matrices along s on the host (csrc/dwf_smat.h) without a GPU, compiled with g++ into a
small program that prints what it builds: which recurrence tables a system gets, and how they
act."""
import os
import subprocess

import numpy as np
import pytest

from paper_1101_0423_gb300 import inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1101_0423_gb300", "csrc")
KINDS = ["M5", "M5T", "S1", "S2", "W", "Z", "ID", "MASS"]

# reads systems (Ns m0 mq, omegas, sigmas) from stdin; prints per system whether it is accepted,
# then per matrix its table's length, whether it is tight, and the table's columns (rows of u for
# unit vectors v, per chirality) and the dense matrix; and for the matrices with a solve the
# errors of the dense rows and of the table on random vectors
PROG = r'''
#include <cstdio>
#include "dwf_smat.h"
using namespace dwf;
typedef long double X;
// M5, M5^T, S1 or S2 (chirality chi) from Eq. 4, 8 and 9 in extended precision, row-major: the
// cyclic system is solved by elimination along s, column by column
static std::vector<X> exact(const SMatrices &m, int kind, int chi) {
  const int n = m.Ns;
  const X kappa = -(X)m.mq / (2 * (X)m.m0), dm = 4 - (X)m.m0;
  std::vector<X> M(n * n), w(n), a(n), b(n), z(n), f(n), g(n);
  for (int s = 0; s < n; ++s) {
    w[s] = sqrtl((X)m.omega[s]);
    a[s] = kind == MK_S2 ? 1 : dm * w[s] + 1 / w[s];
    b[s] = kind == MK_S2 ? (X)m.sigma[s] / m.omega[s] : (dm * m.sigma[s] - 1) / w[s];
  }
  auto at = [&](int j) { return chi ? n - 1 - j : j; };
  for (int t = 0; t < n; ++t) {
    for (int j = 0; j < n; ++j) {  // z_j = f_j + g_j kappa z_last
      const int s = at(j);
      f[j] = ((s == t) - (j ? b[s] * f[j - 1] : 0)) / a[s];
      g[j] = -b[s] / a[s] * (j ? g[j - 1] : 1);
    }
    const X last = f[n - 1] / (1 - g[n - 1] * kappa);
    for (int j = 0; j < n; ++j) z[j] = f[j] + g[j] * kappa * last;
    for (int j = 0; j < n; ++j) {
      const int s = at(j);
      const X u = kind == MK_S2 ? z[j] / w[t] : w[s] * (z[j] + (X)m.sigma[s] / m.omega[s] * (j ? z[j - 1] : kappa * z[n - 1]));
      M[kind == MK_M5T ? t * n + s : s * n + t] = kind == MK_S1 ? u / w[t] : u;
    }
  }
  return M;
}
static unsigned long long seed = 1;
static double rnd() {  // sum of twelve uniforms, less six
  double x = -6;
  for (int i = 0; i < 12; ++i) x += ((seed = seed * 6364136223846793005ull + 1442695040888963407ull) >> 11) * 0x1p-53;
  return x;
}
int main() {
  SMatrices m;
  while (scanf("%d %lf %lf", &m.Ns, &m.m0, &m.mq) == 3) {
    const int n = m.Ns;
    m.omega.resize(n), m.sigma.resize(n);
    for (double &x : m.omega) if (scanf("%lf", &x) != 1) return 1;
    for (double &x : m.sigma) if (scanf("%lf", &x) != 1) return 1;
    const bool ok = build_matrices(&m) && build_recurrences(&m);
    printf("system %d\n", (int)ok);
    if (!ok) continue;
    std::vector<double> v(n), u(n);
    for (int k = 0; k < MK_COUNT; ++k) {
      printf("table %zu %d\n", m.rec[k].size(), (int)m.rec_tight[k]);
      for (int chi = 0; chi < 2; ++chi)
        for (int t = 0; t < n; ++t) {
          std::fill(v.begin(), v.end(), 0.0);
          v[t] = 1.0;
          std::fill(u.begin(), u.end(), 0.0);
          if (!m.rec[k].empty())
            apply_recurrence(m.rec[k].data() + (size_t)chi * n * RC_N, n, (chi ^ (k == MK_M5T)) != 0, v.data(),
                             u.data());
          for (int s = 0; s < n; ++s) printf("%.17g %.17g ", u[s], m.mat[k][(size_t)chi * n * n + s * n + t]);
          printf("\n");
        }
      double ed = 0, er = 0, nn = 0;  // dense rows, table; result
      for (int chi = 0; k < MK_W && chi < 2; ++chi) {
        const std::vector<X> M = exact(m, k, chi);
        const double *D = m.mat[k].data() + (size_t)chi * n * n;
        for (int it = 0; it < 4000 / n + 40; ++it) {
          for (double &x : v) x = rnd();
          if (!m.rec[k].empty())
            apply_recurrence(m.rec[k].data() + (size_t)chi * n * RC_N, n, (chi ^ (k == MK_M5T)) != 0, v.data(), u.data());
          for (int s = 0; s < n; ++s) {
            X want = 0;
            double o = 0;
            for (int t = 0; t < n; ++t) {
              want += M[s * n + t] * v[t];
              o = fma(D[s * n + t], v[t], o);
            }
            nn += (double)(want * want);
            ed += (double)((o - want) * (o - want));
            er += (double)((u[s] - want) * (u[s] - want));
          }
        }
      }
      printf("errors %.6g %.6g\n", sqrt(ed / nn), sqrt(er / nn));
    }
  }
  return 0;
}
'''


@pytest.fixture(scope="module")
def smat(tmp_path_factory):
    d = tmp_path_factory.mktemp("smat")
    src, exe = d / "t.cpp", d / "t"
    src.write_text(PROG)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)])

    def run(ns, m0, mq, om, sg):
        """None if refused, else {kind: (table length, tight, recurrence, dense)}, matrices [chi][s][t]."""
        text = " ".join(repr(float(x)) for x in [m0, mq, *om, *sg])
        lines = iter(subprocess.run([str(exe)], input=f"{ns} {text}\n", text=True, capture_output=True,
                                    check=True).stdout.splitlines())
        if next(lines) == "system 0":
            return None
        out, errors = {}, {}
        for kind in KINDS:
            length, tight = next(lines).split()[1:]
            cols = np.array([[float(x) for x in next(lines).split()] for _ in range(2 * ns)]).reshape(2, ns, ns, 2)
            out[kind] = (int(length), tight == "1", cols[..., 0].transpose(0, 2, 1), cols[..., 1].transpose(0, 2, 1))
            errors[kind] = [float(x) for x in next(lines).split()[1:]]
        out["errors"] = errors
        return out

    return run


@pytest.mark.parametrize("ns,m0,mq,sigma", [(8, 1.8, 500.0, 1 / 2.2), (8, 1e-3, 1.0, 1 / 3.999), (16, 1e-6, 1.0, 0.25),
                                            (5, 1.9, 0.0, 1.0), (64, 1e-3, 30.0, 0.3), (1, 1.8, 500.0, 1 / 2.2)])
def test_bidiagonal_matrices_have_tables_for_every_mass(smat, ns, m0, mq, sigma):
    """omega + sigma L, (d - m0)(omega + sigma L) + 1 - L, 1 and d - m0 are their tables' own
    entries: each has a table, even where the dense corner (d - m0) sigma kappa - kappa loses all
    its digits, and the table gives the exact entries to a few roundings of each."""
    got = smat(ns, m0, mq, np.ones(ns), sigma * np.ones(ns))
    assert got is not None
    dm, kappa = 4.0 - m0, -mq / (2.0 * m0)
    for chi in range(2):
        L = np.diag(np.ones(ns - 1), -1)
        L[0, -1] += kappa
        L = L if chi == 0 else L.T
        want = {"W": np.eye(ns) + sigma * L, "Z": (dm + 1.0) * np.eye(ns) + (dm * sigma - 1.0) * L, "ID": np.eye(ns),
                "MASS": dm * np.eye(ns)}
        for kind, w in want.items():
            length, tight, rec, _ = got[kind]
            assert length and tight
            assert (np.abs(rec[chi] - w) <= 1e-15 * np.abs(w) + 4e-16 * (kind == "Z") * np.abs(L)).all(), kind


@pytest.mark.parametrize("weights", ["shamir", "borici", "cosine"])
@pytest.mark.parametrize("ns", [1, 2, 3, 4, 5, 6, 7, 8, 12, 13, 16, 24, 33, 64])
def test_tables_err_no_more_than_the_dense_rows(smat, weights, ns):
    """Every matrix of the usual weights has a tight table, and applied to random vectors its
    error against extended precision is below that of the dense rows (equal for a single slice;
    S2's (1 + cL)^{-1}, whose factor along s is 1 where sigma = omega, adds as many terms of one
    size as they do: within the scatter of its own few roundings, a third)."""
    got = smat(ns, 1.8, 0.05, *inputs.weights(weights, ns))
    for kind in KINDS:
        assert got[kind][0] == 2 * ns * 4 and got[kind][1], kind
    for kind in ("M5", "M5T", "S1", "S2"):
        dense, table = got["errors"][kind]
        assert table <= (1.34 if kind == "S2" else 1.0) * dense, (kind, dense, table)


@pytest.mark.parametrize("ns,ratio,loose", [(16, 3.0, "M5 M5T S1 S2"), (32, 2.4, "M5 M5T S1 S2"), (16, 1.8, "S2"),
                                            (8, 1.8, "S2"), (16, 1.0, ""), (12, -1.0, "")])
def test_tables_that_grow_along_s_are_not_tight(smat, ns, ratio, loose):
    """Where sigma > omega lets y_0's rounding grow along s beyond the rows' own, the s-mixing
    kernel takes the dense rows; sigma = - omega, where M5 is diagonal, has tables as well."""
    got = smat(ns, 1.8, 0.05, np.ones(ns), ratio * np.ones(ns))
    assert [k for k in KINDS if not got[k][1]] == loose.split()
    for kind in ("M5", "M5T", "S1", "S2"):
        dense, table = got["errors"][kind]
        assert not got[kind][1] or table <= 1.02 * dense
        # the hop epilogue keeps the loose table of M5 and M5^T: within 2.5 of the rows' error
        assert kind not in ("M5", "M5T") or table <= max(2.5 * dense, 2.3e-16)
