"""The FP64 hop's fixed-point products (dwf_device.cuh) where the exponents matter: fields whose
sites differ by many powers of ten, values at the ends of the FP64 range, values that are not
finite, and links that are not SU(3) (the kernels then take plain FP64 arithmetic).

Tolerance: each output real of D^EO is a sum over eight neighbours of products with links.
FP64 arithmetic in any order keeps it within 8 * 12 roundings of 2^-53 times the largest
neighbour (times the link's norm), and the fixed-point form's truncation is below that: 1e-14
of the largest neighbouring |psi| (about 90 * 1.1e-16), times the largest link row norm.
"""
from fractions import Fraction

import numpy as np
import pytest

import oracle
from paper_1101_0423_gb300 import inputs

pytestmark = pytest.mark.gpu
DIMS, NS = (4, 6, 4, 2), 6


def neighbour_max(x):
    """max |psi| over the eight neighbours of each site, per s (shape V4, Ns)."""
    d = DIMS
    m = np.abs(x.reshape(d[3], d[2], d[1], d[0], NS, 24)).max(-1)
    out = np.zeros_like(m)
    for ax in range(4):
        out = np.maximum(out, np.maximum(np.roll(m, 1, ax), np.roll(m, -1, ax)))
    return out.reshape(-1, NS)


def run(dwf, U, x):
    om, sg = inputs.weights("shamir", NS)
    with dwf.Context(DIMS, NS, 1.8, 0.05, om, sg, U) as ctx:
        return dwf.dwf_apply_eo(ctx.h, dwf.OP_DEO, dwf.PREC_F64, 0, x).reshape(-1, NS, 24)


def check(dwf, U, x, link=1.0):
    got, want = run(dwf, U, x), oracle.hop(DIMS, NS, U, 0, x).reshape(-1, NS, 24)
    bound = 1e-14 * link * neighbour_max(x)[..., None] + 5e-324
    on = inputs.site_parity(DIMS) == 0
    assert (np.abs(got - want) <= bound)[on].all(), np.max((np.abs(got - want) / bound)[on])
    assert not got[~on].any()


@pytest.mark.parametrize("decades", [0, 3, 30, 250])
def test_sites_of_different_size(gpu_lib, decades):
    U = inputs.gauge_field(DIMS, 0.5, seed=51)
    x = inputs.gaussian_source(DIMS, NS, seed=52).reshape(-1, NS, 24)
    rng = np.random.RandomState(decades)
    x = x * 10.0 ** rng.uniform(-decades, decades, size=(x.shape[0], NS, 1))
    check(gpu_lib, U, np.ascontiguousarray(x).reshape(-1))


@pytest.mark.parametrize("scale", [1e-320, 1e-308, 1e-290, 1e-284, 1e150, 1e290, 1e306])
def test_ends_of_the_range(gpu_lib, scale):
    U = inputs.gauge_field(DIMS, 0.5, seed=53)
    x = inputs.gaussian_source(DIMS, NS, seed=54) * scale
    got, want = run(gpu_lib, U, x), oracle.hop(DIMS, NS, U, 0, x).reshape(-1, NS, 24)
    bound = 1e-14 * neighbour_max(x)[..., None] + 200 * 5e-324  # denormal results: absolute roundings
    assert (np.abs(got - want) <= bound).all()


def test_links_that_are_not_unitary(gpu_lib):
    U = inputs.gauge_field(DIMS, 0.5, seed=55).reshape(-1, 18)
    U[::7] *= 1.003   # inside the checked bound
    U[3::11] *= 40.0  # outside it
    U[5::13] *= 1e-5
    x = inputs.gaussian_source(DIMS, NS, seed=56)
    check(gpu_lib, U.reshape(-1), x, link=40.0)
    check(gpu_lib, np.zeros_like(U).reshape(-1), x)


def test_values_that_are_not_finite(gpu_lib):
    """A NaN or an infinity reaches the outputs that its spin projections enter (h_j of Eq. 12
    for each direction, all colours), and no others: those are as with a zero in its place."""
    U = inputs.gauge_field(DIMS, 0.5, seed=57)
    x = inputs.gaussian_source(DIMS, NS, seed=58).reshape(-1, NS, 24)
    odd = np.flatnonzero(inputs.site_parity(DIMS) == 1)
    nx, ny, nz, nt = DIMS
    expect = np.zeros((nt, nz, ny, nx, NS, 4), bool)
    for site, s, c, v in ((odd[3], 1, 5, np.nan), (odd[40], 4, 17, np.inf), (odd[77], 0, 20, -np.inf)):
        x[site, s, c] = v
        at = [site // (nx * ny * nz), site // (nx * ny) % nz, site // nx % ny, site % nx]
        spin = c // 6
        for mu in range(4):
            j = spin if spin < 2 else (1 - (spin - 2) if mu < 2 else spin - 2)
            for step in (1, -1):
                to = list(at)
                to[3 - mu] = (to[3 - mu] + step) % DIMS[mu]
                expect[tuple(to) + (s, j)] = True
                expect[tuple(to) + (s, 2 + (1 - j if mu < 2 else j))] = True
    got = run(gpu_lib, U, x.reshape(-1))
    bad = np.repeat(expect.reshape(-1, NS, 4), 6, axis=2)
    assert np.array_equal(~np.isfinite(got), bad)
    clean = np.where(np.isfinite(x), x, 0.0).reshape(-1)
    want = oracle.hop(DIMS, NS, U, 0, clean).reshape(-1, NS, 24)
    bound = 1e-14 * neighbour_max(clean)[..., None]
    assert (np.abs(got - want) <= bound)[~bad].all()


def exact_m5(ns, m0, mq, ratio):
    """M5 of Eq. 8 per chirality for omega = 1, sigma = ratio, column by column in rationals: u = (1 +
    cL) z with (a + b L) z = v, a = (d - m0) + 1, b = (d - m0) sigma - 1, and kappa = L's corner."""
    F = Fraction
    kappa, dm, sg = -F(mq) / (2 * F(m0)), 4 - F(m0), F(ratio)
    a, b = dm + 1, dm * sg - 1
    M = np.empty((ns, ns), dtype=object)
    for t in range(ns):
        f, g, fs, gs = F(0), F(1), [], []
        for j in range(ns):
            f, g = (F(int(j == t)) - b * f) / a, -b * g / a
            fs.append(f), gs.append(g)
        zl = fs[-1] / (1 - gs[-1] * kappa)
        z = [x + y * kappa * zl for x, y in zip(fs, gs)]
        for j in range(ns):
            M[j, t] = z[j] + sg * (z[j - 1] if j else kappa * z[-1])
    M = M.astype(float)
    return M, M[::-1, ::-1].copy()  # chirality -: L^T, which runs the other way


def rows_error(ns, m0, mq, ratio):
    """Bound of the relative error of M5's rows and tables for omega = 1: a rounding made in the
    solve along s comes round through the corner |kappa| grown by ((d - m0) sigma - 1) / ((d - m0)
    + 1) a step where that is above 1, with Ns of them (45 roundings of the products besides)."""
    grow = max(1.0, ((4 - m0) * ratio - 1) / (5 - m0)) ** ns
    return 45 * 2.3e-16 + ns * 2.3e-16 * (grow - 1) * max(mq / (2 * m0), 1e-3)


@pytest.mark.parametrize("opname", ["M5", "M5T", "C", "CDAG", "CCDAG", "DFULL"])
@pytest.mark.parametrize("ns,ratio", [(1, 1.0), (2, 0.0), (7, 1.0), (16, 1.0), (33, 0.5), (64, 1.0), (16, 1.8),
                                      (16, -1.0), (16, 3.0), (32, 2.4)])
def test_matrices_along_s(gpu_lib, opname, ns, ratio):
    """The FP64 matrices along s as recurrences and, where sigma > omega lets the closure's
    rounding grow along s (3.0 at Ns = 16, 2.4 at 32: test_smat_host.py), as dense rows in the
    s-mixing kernel; the hop epilogues keep the recurrence.  M5 against exact rationals, each
    M5 within rows_error of the field's and the matrix's size, each hop a factor of at most 8."""
    dwf, dims, m0, mq = gpu_lib, (2, 4, 2, 6), 1.8, 0.05
    om, sg = np.ones(ns), ratio * np.ones(ns)
    U = inputs.gauge_field(dims, 0.5, seed=60)
    x = inputs.gaussian_source(dims, ns, seed=61)
    mp, mm = exact_m5(ns, m0, mq, ratio)
    with dwf.Context(dims, ns, m0, mq, om, sg, U) as ctx:
        got = dwf.dwf_apply_eo(ctx.h, getattr(dwf, "OP_" + opname), dwf.PREC_F64, 1, x)
    tol = rows_error(ns, m0, mq, ratio)
    if opname == "DFULL":
        want, tol = oracle.dfull(dims, ns, U, m0, mq, om, sg, x), 45 * 2.3e-16
    elif opname in ("M5", "M5T"):
        want = oracle.apply_s(dims, ns, mp, mm, x, transpose=opname == "M5T", parity=1)
    else:
        # |out| of one hop and M5 pair is within 4 |M5| of its input: errors of both add up
        want = {"C": oracle.c_op, "CDAG": oracle.cdag_op, "CCDAG": oracle.ccdag_op}[opname](dims, ns, U, mp, mm, 1, x)
        m5 = max(1.0, np.abs(mp).sum(1).max())
        tol *= 4 * (4 * m5) ** (4 if opname == "CCDAG" else 2) * np.abs(x).max() / np.abs(want).max()
    assert np.abs(got - want).max() <= tol * max(1.0, np.abs(want).max())


def test_solve_where_the_matrices_along_s_are_dense(gpu_lib):
    """A full solve whose reconstruction takes the dense S2 (sigma = 1.8 omega, Ns = 8)."""
    dwf, dims, ns, m0, mq = gpu_lib, (4, 4, 2, 4), 8, 1.8, 0.1
    om, sg = np.ones(ns), 1.8 * np.ones(ns)
    U = inputs.gauge_field(dims, 0.3, seed=64)
    eta = inputs.gaussian_source(dims, ns, seed=65)
    with dwf.Context(dims, ns, m0, mq, om, sg, U) as ctx:
        psi, st = dwf.dwf_solve(ctx.h, eta, tol=1e-10)
    res = np.linalg.norm(eta - oracle.dfull(dims, ns, U, m0, mq, om, sg, psi)) / np.linalg.norm(eta)
    assert st["converged"] == 1 and res <= 1e-10


def test_whole_operator_where_the_dense_corner_cancels(gpu_lib):
    """D(mq) in FP64 for a mass and weights at which (d - m0) sigma is 1 to three digits and the
    corner |kappa| = 500: the bidiagonal matrices come from their tables (the dense Z agrees with
    its own to 5e-14 only).  Each output is a sum of products whose largest, |kappa| |psi| and
    sigma |kappa| |H psi|, cancel to 1e-3 of themselves at worst: within 100 of their roundings."""
    dwf, dims, ns, m0, mq = gpu_lib, (2, 4, 2, 6), 8, 1e-3, 1.0
    om, sg = np.ones(ns), np.ones(ns) / 3.999
    U = inputs.gauge_field(dims, 0.5, seed=62)
    x = inputs.gaussian_source(dims, ns, seed=63)
    with dwf.Context(dims, ns, m0, mq, om, sg, U) as ctx:
        got = dwf.dwf_apply_eo(ctx.h, dwf.OP_DFULL, dwf.PREC_F64, 1, x)
    want = oracle.dfull(dims, ns, U, m0, mq, om, sg, x)
    assert np.abs(got - want).max() <= 100 * 1.2e-16 * 500 * np.abs(x).max()


def test_link_out_of_bounds_changes_its_own_sites_only(gpu_lib):
    """Which arithmetic a site takes depends on its own links: one link scaled out of the checked
    bound leaves every output but those at its two ends bit for bit as it was, whatever tile
    they share with them."""
    U = inputs.gauge_field(DIMS, 0.5, seed=66).reshape(-1, 4, 18)
    x = inputs.gaussian_source(DIMS, NS, seed=67)
    before = run(gpu_lib, U.reshape(-1), x)
    nx, ny, nz, nt = DIMS
    for site, mu in ((0, 0), (nx * ny * nz + 5, 3), (37, 1)):
        V = U.copy()
        V[site, mu] *= 40.0
        at = [site % nx, site // nx % ny, site // (nx * ny) % nz, site // (nx * ny * nz)]
        at[mu] = (at[mu] + 1) % DIMS[mu]
        ends = {site, at[0] + nx * (at[1] + ny * (at[2] + nz * at[3]))}
        differ = set(np.flatnonzero((run(gpu_lib, V.reshape(-1), x) != before).any((1, 2))))
        assert differ == {e for e in ends if inputs.site_parity(DIMS)[e] == 0}


def hop_terms(U, x):
    """Sizes of the terms of D^EO, sum_mu sum_b |U_ab| |h_b| over the eight hops, per complex component
    (V4, Ns, 4, 3): h = psi_up -+ A psi_dn with A = -i sigma_k, 1 (chiral basis), and the lower spins
    A^dag of the same products."""
    A = [np.array(m) for m in ([[0, -1j], [-1j, 0]], [[0, -1], [1, 0]], [[-1j, 0], [0, 1j]], [[1, 0], [0, 1]])]
    nx, ny, nz, nt = DIMS
    psi = np.ascontiguousarray(x).view(np.complex128).reshape(nt, nz, ny, nx, NS, 4, 3)
    W = np.abs(U.view(np.complex128).reshape(nt, nz, ny, nx, 4, 3, 3))
    S = np.zeros(psi.shape)
    for mu in range(4):
        ax = 3 - mu
        for sign, step in ((-1, -1), (1, 1)):
            p = np.roll(psi, step, ax)
            h = np.abs(p[..., :2, :] + sign * np.einsum("jk,...kc->...jc", A[mu], p[..., 2:, :]))
            w = W[..., mu, :, :] if sign < 0 else np.swapaxes(np.roll(W[..., mu, :, :], 1, ax), -1, -2)
            t = np.einsum("tzyxab,tzyxsjb->tzyxsja", w, h)
            S[..., :2, :] += t
            S[..., 2:, :] += np.einsum("kj,...ja->...ka", np.abs(A[mu]).T, t)
    return 0.5 * S.reshape(-1, NS, 4, 3)


@pytest.mark.parametrize("decades", [0, 3, 9, 18, 40])
@pytest.mark.parametrize("links", ["unit", "diagonal", "nearly unit", "SU(3)", "one size a link"])
def test_components_of_different_size(gpu_lib, links, decades):
    """Every complex component of D^EO to FP64 accuracy relative to its own terms, whatever the
    sizes of the field's other colours and spins, where the links mix them and where they do
    not.  Bound: 84 units at worst (ten and a half a hop) against 2^51 of the component's terms,
    3.8e-14 of them; the root mean square of the errors is that of FP64 roundings."""
    rng = np.random.RandomState(decades + 1)
    n = int(np.prod(DIMS)) * 4
    if links in ("unit", "diagonal", "one size a link"):
        ph = rng.uniform(0, 2 * np.pi, (n, 3)) * (links != "unit")
        ph[:, 2] = -ph[:, 0] - ph[:, 1]
        size = 10.0 ** rng.uniform(-decades, 0, (n, 1)) if links == "one size a link" else 1.0
        U = np.ascontiguousarray((np.exp(1j * ph) * size)[:, :, None] * np.eye(3)).view(float).reshape(-1)
    else:
        U = inputs.gauge_field(DIMS, 0.5 if links == "SU(3)" else 1e-9, seed=68)
    x = inputs.gaussian_source(DIMS, NS, seed=69).reshape(-1, NS, 12, 2)
    x = np.ascontiguousarray(x * 10.0 ** rng.uniform(-decades, 0, (x.shape[0] if decades == 9 else 1, NS, 12, 1)))
    got, want = run(gpu_lib, U, x.reshape(-1)), oracle.hop(DIMS, NS, U, 0, x.reshape(-1)).reshape(-1, NS, 24)
    on = inputs.site_parity(DIMS) == 0
    err = np.abs((got - want).view(np.complex128).reshape(-1, NS, 4, 3))[on]
    rel = err / hop_terms(U, x.reshape(-1))[on]
    print(f"{links} {decades}: max {rel.max():.2e} rms {np.sqrt((rel ** 2).mean()):.2e}")
    assert rel.max() <= 3.8e-14
    assert np.sqrt((rel ** 2).mean()) <= 2.3e-16


def test_components_at_the_smallest_exponent(gpu_lib):
    """Upper spins whose largest component has the smallest exponent of the fixed-point range (2^-943),
    on unit links: the components a billion times smaller keep FP64's accuracy too."""
    U = np.ascontiguousarray(np.broadcast_to(np.eye(3, dtype=complex), (int(np.prod(DIMS)) * 4, 3, 3))).view(float).reshape(-1)
    rng = np.random.RandomState(5)
    x = rng.uniform(1.0, 1.999, (int(np.prod(DIMS)), NS, 12, 2)) * 2.0 ** -943
    x[:, :, 1:6] *= 1e-9
    x[:, :, 6:] = 0.0
    got, want = run(gpu_lib, U, x.reshape(-1)), oracle.hop(DIMS, NS, U, 0, x.reshape(-1)).reshape(-1, NS, 24)
    terms = np.repeat(hop_terms(U, x.reshape(-1)).reshape(-1, NS, 12), 2, axis=2)
    assert (np.abs(got - want) <= 3.8e-14 * terms)[inputs.site_parity(DIMS) == 0].all()


def test_components_without_terms_are_zero(gpu_lib):
    """A field with one spin and colour on links that do not mix colours: every component that no
    term reaches is exactly 0, the others are as in FP64."""
    U = np.ascontiguousarray(np.broadcast_to(np.eye(3, dtype=complex), (int(np.prod(DIMS)) * 4, 3, 3))).view(float).reshape(-1)
    x = inputs.gaussian_source(DIMS, NS, seed=70).reshape(-1, NS, 12, 2)
    x[:, :, np.arange(12) != 4] = 0.0
    got, want = run(gpu_lib, U, x.reshape(-1)), oracle.hop(DIMS, NS, U, 0, x.reshape(-1)).reshape(-1, NS, 24)
    terms = hop_terms(U, x.reshape(-1))
    assert (got.view(np.complex128).reshape(terms.shape)[terms == 0] == 0).all()
    assert (np.abs(got - want).view() <= 4.5e-16 * np.repeat(terms.reshape(-1, NS, 12), 2, axis=2)).all()
