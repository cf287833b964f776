"""The s-mixing kernel's CTA sizes (csrc/dwf_launch.cuh: 128 threads, from Ns = 32, 33 or 48 on 256) on
both sides of each line, against the FP64 CPU oracle: operators in FP32 and bf16 within the
parity tests' tolerances (the 48 half-lattice sites are no multiple of a CTA's 2 to 7), and a
solve whose p-update takes them."""
import numpy as np
import pytest

import oracle
from paper_1101_0423_gb300 import inputs

pytestmark = pytest.mark.gpu
DIMS, M0, MQ = (2, 2, 4, 6), 1.8, 0.08


@pytest.mark.parametrize("ns", [31, 32, 33, 47, 48, 64])
def test_operators_and_solve(gpu_lib, ns):
    dwf = gpu_lib
    om, sg = inputs.weights("borici", ns)
    U = inputs.gauge_field(DIMS, 0.4, seed=91)
    x = inputs.gaussian_source(DIMS, ns, seed=92)
    mp, mm = oracle.m5(ns, M0, MQ, om, sg)
    want = {"M5": oracle.apply_s(DIMS, ns, mp, mm, x, parity=1), "CDAG": oracle.cdag_op(DIMS, ns, U, mp, mm, 1, x),
            "DFULL": oracle.dfull(DIMS, ns, U, M0, MQ, om, sg, x)}
    with dwf.Context(DIMS, ns, M0, MQ, om, sg, U) as ctx:
        for prec, tol in ((dwf.PREC_F32, 1e-5), (dwf.PREC_BF16, 3e-2)):
            for op, w in want.items():
                got = dwf.dwf_apply_eo(ctx.h, getattr(dwf, "OP_" + op), prec, 1, x)
                assert np.max(np.abs(got - w)) <= tol * np.max(np.abs(w)), (op, prec)
        psi, st = dwf.dwf_solve(ctx.h, x, tol=1e-10)
    res = np.linalg.norm(x - oracle.dfull(DIMS, ns, U, M0, MQ, om, sg, psi)) / np.linalg.norm(x)
    assert st["converged"] == 1 and res <= 1e-10
