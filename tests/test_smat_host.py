"""The matrices along s on the host (csrc/dwf_smat.h) without a GPU, compiled with g++ into a
small program that prints what it builds: which recurrence tables a system gets, and how they
act."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1101_0423_gb300", "csrc")
KINDS = ["M5", "M5T", "S1", "S2", "W", "Z", "ID", "MASS"]

# reads systems (Ns m0 mq, omegas, sigmas) from stdin; prints per system whether it is accepted,
# then per matrix its table's length, whether it is tight, and the table's columns (rows of u for
# unit vectors v, per chirality) and the dense matrix
PROG = r'''
#include <cstdio>
#include "dwf_smat.h"
using namespace dwf;
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
            apply_recurrence(m.rec[k].data() + (size_t)chi * n * RC_N, n, (chi ^ (k == MK_M5T)) != 0,
                             -m.mq / (2.0 * m.m0), v.data(), u.data());
          for (int s = 0; s < n; ++s) printf("%.17g %.17g ", u[s], m.mat[k][(size_t)chi * n * n + s * n + t]);
          printf("\n");
        }
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
        out = {}
        for kind in KINDS:
            length, tight = next(lines).split()[1:]
            cols = np.array([[float(x) for x in next(lines).split()] for _ in range(2 * ns)]).reshape(2, ns, ns, 2)
            out[kind] = (int(length), tight == "1", cols[..., 0].transpose(0, 2, 1), cols[..., 1].transpose(0, 2, 1))
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
