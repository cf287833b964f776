"""The work that users of the domain-wall solver have it do, as cases to be timed and compared.

A case calls one public entry point of ``paper_1101_0423_gb300.dwf`` on device arrays, as an
application with its fields on the GPU does:

``op``      ``dwf_apply_eo_dev`` (or ``dwf_apply_eo_dev_static``): one operator on one field
``solve``   ``dwf_solve_dev``: one system to a true relative residual of ``tol``
``ragged``  ``dwf_solve_ragged_dev``: several systems of different Ns and mass on one gauge field
``prop``    ``dwf_load_gauge_dev`` and ``dwf_propagator_dev``: a new configuration of an
            ensemble arrives and its 12-source quark propagator is taken (a batched solve)

Every input is drawn on the GPU from the seed alone: links exp(i eps H) with H a random
traceless Hermitian matrix, complex Gaussian sources.  ``exact`` evaluates the same
definitions (Eq. 1-12 of arXiv:1101.0423) in complex128 with plain torch.
"""
import math

import numpy as np
import torch

from paper_1101_0423_gb300 import dwf, inputs

M0 = 1.8
PRECS = {"f64": dwf.PREC_F64, "f32": dwf.PREC_F32, "f16": dwf.PREC_F16, "bf16": dwf.PREC_BF16}
REAL_BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
OPS = {"DEO": dwf.OP_DEO, "DOE": dwf.OP_DOE, "M5": dwf.OP_M5, "M5T": dwf.OP_M5T, "C": dwf.OP_C,
       "CDAG": dwf.OP_CDAG, "CCDAG": dwf.OP_CCDAG, "DFULL": dwf.OP_DFULL, "DW": dwf.OP_DW}
LARGEST_5D = 24 * 24 * 24 * 48 * 8  # sites x Ns of the largest listed case


def _op(name, op, prec, dims, ns, weights, mq, eps=0.5, parity=1, static=False):
    return dict(name=name, kind="op", op=op, prec=prec, nx=dims[0], ny=dims[1], nz=dims[2], nt=dims[3], ns=ns,
                weights=weights, mq=mq, eps=eps, parity=parity, static=static)


def _solve(name, prec, dims, ns, weights, mq, iters, eps=0.5, parity=1, normal=False):
    return dict(name=name, kind="solve", prec=prec, nx=dims[0], ny=dims[1], nz=dims[2], nt=dims[3], ns=ns,
                weights=weights, mq=mq, iters=iters, eps=eps, parity=parity, normal=normal, tol=1e-10)


def listed():
    return [
        # the smallest call: one hopping block on the 4^4 lattice of the first workload, where
        # launches and waits are everything (an application's own Krylov loop on a test lattice)
        _op("deo_f32_4x4x4x4_ns8", "DEO", "f32", (4, 4, 4, 4), 8, "shamir", 0.05, eps=0.3, parity=0),
        # the allocation-free entry point at the size its static array is for, C in FP32
        _op("static_c_f32_8x8x8x16_ns12", "C", "f32", (8, 8, 8, 16), 12, "borici", 0.05, static=True),
        # odd Ns and extents that fill no tile evenly; the single dslash in FP32
        _op("doe_f32_14x10x6x18_ns5", "DOE", "f32", (14, 10, 6, 18), 5, "cosine", 0.02),
        # 16-bit storage, large Ns (the served workload's second lattice): an inner operator of
        # an outer solver of the application's own
        _op("cdag_bf16_12x12x12x24_ns24", "CDAG", "bf16", (12, 12, 12, 24), 24, "borici", 0.03),
        # the normal operator on the benchmark's lattice, in the inner and in the outer precision
        # (the latter is a true residual of a user's own solver)
        _op("ccdag_f32_16x16x16x32_ns16", "CCDAG", "f32", (16, 16, 16, 32), 16, "cosine", 0.02),
        _op("ccdag_f64_16x16x16x32_ns16", "CCDAG", "f64", (16, 16, 16, 32), 16, "cosine", 0.02),
        # the largest lattice: the whole 5D operator in FP64, which checks a solution
        _op("dfull_f64_24x24x24x48_ns8", "DFULL", "f64", (24, 24, 24, 48), 8, "shamir", 0.01),
        # the first workload: normal equations on a 4^4 lattice, source on the even sites
        _solve("solve_normal_f32_4x4x4x4_ns8", "f32", (4, 4, 4, 4), 8, "shamir", 0.05, 441, eps=0.3, parity=0,
               normal=True),
        # the benchmark: one full solve at 16^3 x 32 x 16
        _solve("solve_f32_16x16x16x32_ns16", "f32", (16, 16, 16, 32), 16, "cosine", 0.02, 1303),
        # a request of the served workload: bf16 inner iterations, library's default mode
        _solve("solve_bf16_12x12x12x24_ns8", "bf16", (12, 12, 12, 24), 8, "borici", 0.05, 800),
        # a set of different Ns and masses on one shared gauge field, solved together
        dict(name="ragged_f32_8x8x8x8_ns8_12_16_24", kind="ragged", prec="f32", nx=8, ny=8, nz=8, nt=8,
             ns_set="8,12,16,24", mq_lo=0.02, mq_hi=0.1, weights="shamir", eps=0.5, iters=800, tol=1e-10),
        # a measurement: new configuration, 12 spin-colour point sources as one batch
        dict(name="prop_f32_8x8x8x8_ns8", kind="prop", prec="f32", nx=8, ny=8, nz=8, nt=8, ns=8, weights="shamir",
             mq=0.05, eps=0.5, iters=600, tol=1e-10),
    ]


def _extents(rng, most):
    """Four even extents with at most `most` sites, their volume spread over its logarithm."""
    want = math.exp(rng.uniform(math.log(4 ** 4), math.log(most)))
    while True:
        side = want ** 0.25
        d = [max(4, 2 * round(side * math.exp(rng.uniform(-0.5, 0.5)) / 2)) for _ in range(4)]
        v = d[0] * d[1] * d[2] * d[3]
        if v <= most and 0.6 * want <= v <= 1.7 * want:
            return d


def draw(rng):
    kind = rng.choice(["op", "op", "op", "op", "solve", "solve", "ragged", "prop"])
    weights = rng.choice(["shamir", "borici", "cosine"])
    mq = math.exp(rng.uniform(math.log(0.01), math.log(0.1)))
    if kind == "op":
        ns = rng.choice([4, 5, 6, 7, 8, 8, 10, 12, 12, 13, 16, 16, 20, 24, 32])
        d = _extents(rng, LARGEST_5D // ns)
        op = rng.choice(["DEO", "DOE", "M5", "M5T", "C", "CDAG", "CCDAG", "CCDAG", "DFULL", "DW"])
        prec = rng.choice(["f64", "f32", "f32", "f16", "bf16"])
        static = (prec == "f32" and op not in ("DFULL", "DW") and d[0] * d[1] * d[2] * d[3] * ns <= 240000
                  and rng.random() < 0.5)
        c = _op("", op, prec, d, ns, weights, mq, parity=rng.randrange(2), static=static)
    elif kind == "solve":
        ns = rng.choice([5, 6, 8, 10, 12, 16, 20, 24])
        d = _extents(rng, min(12 ** 3 * 24, 16 ** 3 * 32 * 4 // ns))
        c = _solve("", rng.choice(["f32", "f32", "bf16"]), d, ns, weights, mq, 60 * ns + 200,
                   parity=rng.randrange(2), normal=rng.random() < 0.3)
    elif kind == "ragged":
        d = _extents(rng, 8 ** 4)
        ns = [rng.choice([5, 8, 10, 12, 16, 20, 24]) for _ in range(rng.choice([2, 3, 4]))]
        c = dict(kind="ragged", prec="f32", nx=d[0], ny=d[1], nz=d[2], nt=d[3], ns_set=",".join(map(str, ns)),
                 mq_lo=0.02, mq_hi=mq + 0.02, weights=weights, eps=0.5, iters=800, tol=1e-10)
    else:
        d = _extents(rng, 8 ** 4)
        c = dict(kind="prop", prec="f32", nx=d[0], ny=d[1], nz=d[2], nt=d[3], ns=rng.choice([4, 6, 8, 10, 12]),
                 weights=weights, mq=mq, eps=0.5, iters=600, tol=1e-10)
    c.pop("name", None)
    return c


# ---------------------------------------------------------------- inputs

def _dims(case):
    return case["nx"], case["ny"], case["nz"], case["nt"]


def _gen(seed, tag):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + tag)
    return g


def _gauge(dims, eps, seed):
    """U_mu(x) = exp(i eps H) in the host layout, FP64 on the GPU."""
    n = inputs.volume(dims) * 4
    a = torch.randn(n, 3, 3, 2, generator=_gen(seed, 1), device="cuda", dtype=torch.float64)
    a = torch.view_as_complex(a)
    h = 0.5 * (a + a.mH)
    h = h - (h.diagonal(dim1=-2, dim2=-1).sum(-1).real / 3.0)[:, None, None] * torch.eye(3, device="cuda")
    return torch.view_as_real(torch.linalg.matrix_exp(1j * eps * h)).reshape(-1).contiguous()


def _source(dims, ns, seed, tag=2, parity=None):
    x = torch.randn(inputs.volume(dims), ns * 24, generator=_gen(seed, tag), device="cuda", dtype=torch.float64)
    if parity is not None:
        x[torch.from_numpy(inputs.site_parity(dims) != parity).cuda()] = 0.0
    return x.reshape(-1)


def _masses(case):
    """(Ns, mq) of the members of a ragged set: masses spread evenly over their logarithm."""
    ns = [int(v) for v in case["ns_set"].split(",")]
    f = np.linspace(0.0, 1.0, len(ns))
    return [(n, float(case["mq_lo"] * (case["mq_hi"] / case["mq_lo"]) ** x)) for n, x in zip(ns, f)]


def _context(case, ns, mq):
    om, sg = inputs.weights(case["weights"], ns)
    return dwf.Context(_dims(case), ns, M0, mq, om, sg)


def prepare(case, seed):
    dims, kind = _dims(case), case["kind"]
    U = _gauge(dims, case["eps"], seed)
    st = {"case": case, "stream": torch.cuda.current_stream()}
    if kind == "ragged":
        torch.cuda.synchronize()
        gauge = dwf.dwf_gauge_create_dev(dims, U, stream=st["stream"])
        members = _masses(case)
        st["ctx"] = [_context(case, ns, mq) for ns, mq in members]
        for c in st["ctx"]:
            dwf.dwf_attach_gauge(c.h, gauge)
        dwf.dwf_gauge_release(gauge)  # the contexts keep it
        st["rhs"] = [_source(dims, ns, seed, tag=2 + k) for k, (ns, _) in enumerate(members)]
        st["sol"] = [torch.empty_like(x) for x in st["rhs"]]
        return st
    st["ctx"] = _context(case, case["ns"], case["mq"])
    if kind == "prop":
        st["U"] = U
        st["x0"] = [int(v) for v in np.random.RandomState(int(seed) & 0x7FFFFFFF).randint(0, dims)]
        st["prop"] = torch.empty(inputs.volume(dims) * 144 * 2, device="cuda", dtype=torch.float64)
        return st
    torch.cuda.synchronize()
    dwf.dwf_load_gauge_dev(st["ctx"].h, U, stream=st["stream"])
    on = case["parity"] if kind == "solve" and case["normal"] else None
    st["rhs"] = _source(dims, case["ns"], seed, parity=on)
    st["sol"] = torch.empty_like(st["rhs"])
    return st


def run(state):
    case, s = state["case"], state["stream"]
    kind = case["kind"]
    if kind == "op":
        f = dwf.dwf_apply_eo_dev_static if case["static"] else dwf.dwf_apply_eo_dev
        f(state["ctx"].h, OPS[case["op"]], PRECS[case["prec"]], case["parity"], state["rhs"], state["sol"], stream=s)
        return state["sol"]
    kw = dict(tol=case["tol"], inner_prec=PRECS[case["prec"]])
    if kind == "solve":
        dwf.dwf_solve_dev(state["ctx"].h, state["rhs"], state["sol"], stream=s, schur_parity=case["parity"],
                          system=dwf.SYS_NORMAL if case["normal"] else dwf.SYS_FULL, **kw)
        return state["sol"]
    if kind == "ragged":
        dwf.dwf_solve_ragged_dev([c.h for c in state["ctx"]], state["rhs"], state["sol"], stream=s, **kw)
        return state["sol"]
    dwf.dwf_load_gauge_dev(state["ctx"].h, state["U"], stream=s)
    _propagator_dev(state["ctx"].h, state["x0"], state["prop"], s, kw)
    return state["prop"]


def _propagator_dev(ctx, x0, d_prop, stream, kw):
    """dwf_propagator_dev through the library's own signature (the binding wraps the host form)."""
    import ctypes
    p = dwf.dwf_solve_params_default()
    for k, v in kw.items():
        setattr(p, k, v)
    stats = (dwf.SolveStats * 12)()
    rc = dwf.load().dwf_propagator_dev(ctx, (ctypes.c_int * 4)(*x0), ctypes.byref(p), d_prop.data_ptr(), stats,
                                       stream.cuda_stream)
    if rc != dwf.DWF_OK:
        raise dwf.DwfError(rc, dwf.dwf_last_error(ctx))


# ---------------------------------------------------------------- work, tolerance

HOP = 1320.0  # flops of the hopping term per 5D site


def _m5_flops(ns):
    """M5 along s, per 5D site: the cyclic bidiagonal solve and product of Eq. 8 (about six
    fused multiply-adds per real)."""
    return 24.0 * min(2 * ns - 1, 12)


def work(case):
    """Bytes: sources or input field read and result written once, links read once.  Flops: the
    operator's hops and M5s on the sites they act on; a solve's iterations (measured counts for
    the listed cases, a rule of thumb for drawn ones) at two operators and six vector
    operations each."""
    v4 = inputs.volume(_dims(case))
    rb = REAL_BYTES[case["prec"]]
    links = v4 * 4 * 18.0 * (rb if rb >= 4 else rb * 12 / 18)
    if case["kind"] == "op":
        ns = case["ns"]
        n, op, m5 = v4 * ns, case["op"], _m5_flops(ns)
        half = {"DEO": HOP, "DOE": HOP, "M5": m5, "M5T": m5, "C": 2 * (HOP + m5) + 48, "CDAG": 2 * (HOP + m5) + 48,
                "CCDAG": 4 * (HOP + m5) + 96}
        if op in ("M5", "M5T"):
            links = 0.0
        if op in half:  # one parity in, the whole (half zero) lattice out
            return {"bytes": n * 192.0 * 1.5 + links, "flops": 0.5 * n * half[op]}
        s_work = 48.0 + (96.0 if op == "DFULL" else 0.0)
        return {"bytes": n * 192.0 * 2 + links, "flops": n * (HOP + s_work)}
    if case["kind"] == "ragged":
        sets, rows = _masses(case), 1
    else:
        sets, rows = [(case["ns"], case["mq"])], 12 if case["kind"] == "prop" else 1
    total = {"bytes": links, "flops": 0.0}
    for ns, _ in sets:
        n = v4 * ns
        total["flops"] += rows * case["iters"] * 0.5 * n * (4 * (HOP + _m5_flops(ns)) + 240)
        total["bytes"] += rows * n * 192.0 * 2 if case["kind"] != "prop" else 0.0
    if case["kind"] == "prop":
        total["bytes"] += v4 * 144 * 16.0
    return total


def tolerance(case):
    """About four times what the path shows against ``exact`` in its own precision."""
    if case["kind"] == "op":
        # roundings of the storage precision, through one to four hops and M5 applications
        return {"f64": {"rel": 2e-15, "max": 4e-14}, "f32": {"rel": 5e-7, "max": 1e-5},
                "f16": {"rel": 1.5e-3, "max": 2e-2}, "bf16": {"rel": 1e-2, "max": 0.15}}[case["prec"]]
    # two solutions of the same system, each with a true relative residual of at most 1e-10,
    # differ by up to that times the system's conditioning
    return {"rel": 5e-9, "max": 1e-6}


# ---------------------------------------------------------------- the same in complex128 torch

def _gammas():
    s = [np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]], complex)]
    z = np.zeros((2, 2))
    g = [np.block([[z, -1j * m], [1j * m, z]]) for m in s] + [np.block([[z, np.eye(2)], [np.eye(2), z]])]
    return [torch.from_numpy(np.ascontiguousarray(m, dtype=complex)).cuda() for m in g]


class _Exact:
    """Eq. 1-12 on full-lattice fields [..., t, z, y, x, s, spin, colour] in complex128."""

    def __init__(self, dims, ns, mq, weights, U):
        self.dims, self.ns = dims, ns
        self.U = torch.view_as_complex(U.reshape(-1, 2)).reshape(dims[3], dims[2], dims[1], dims[0], 4, 3, 3)
        self.g = _gammas()
        om, sg = inputs.weights(weights, ns)
        lp = np.zeros((ns, ns))
        for s in range(1, ns):
            lp[s, s - 1] = 1.0
        lp[0, ns - 1] = -mq / (2.0 * M0)
        dm, one = 4.0 - M0, np.eye(ns)
        self.W, self.M5, self.L1, self.S1, self.S2 = [], [], [], [], []
        for L in (lp, lp.T):
            w = np.diag(om) + np.diag(sg) @ L
            y = one + np.diag(sg / om) @ L
            rs = np.diag(1.0 / np.sqrt(om))
            m5 = np.linalg.inv(dm * one + rs @ (one - L) @ np.linalg.inv(y) @ rs)
            self.W.append(w)
            self.L1.append(one - L)
            self.M5.append(m5)
            self.S1.append(m5 @ rs)
            self.S2.append(np.linalg.inv(y) @ rs)
        par = torch.from_numpy(inputs.site_parity(dims)).cuda().reshape(dims[3], dims[2], dims[1], dims[0])
        self.mask = [(par == p).to(torch.float64)[..., None, None, None] for p in (0, 1)]

    def field(self, x):
        d = self.dims
        return torch.view_as_complex(x.reshape(-1, 2)).reshape(d[3], d[2], d[1], d[0], self.ns, 4, 3)

    def hop(self, psi):
        """-1/2 sum_mu [(1 - g_mu) U_mu(x) psi(x+mu) + (1 + g_mu) U_mu(x-mu)^dag psi(x-mu)]"""
        out = torch.zeros_like(psi)
        for mu in range(4):
            ax = -4 - mu
            u = self.U[..., mu, :, :]
            # [site, s * spin, colour] x [site, colour, colour]
            shape = psi.shape
            fwd = torch.roll(psi, -1, dims=ax).flatten(-3, -2)
            fwd = torch.matmul(fwd, u.transpose(-1, -2)).reshape(shape)
            bwd = torch.matmul(psi.flatten(-3, -2), u.conj()).reshape(shape)
            bwd = torch.roll(bwd, 1, dims=ax)
            out += fwd + bwd
            d = bwd - fwd
            out += torch.matmul(self.g[mu], d)
        return -0.5 * out

    def along_s(self, mats, psi, transpose=False):
        out = torch.empty_like(psi)
        for chi in (0, 1):
            m = torch.from_numpy(np.ascontiguousarray(mats[chi].T if transpose else mats[chi])).cuda()
            part = psi[..., 2 * chi:2 * chi + 2, :].flatten(-2)
            part = torch.view_as_real(part).flatten(-2)
            part = torch.view_as_complex(torch.matmul(m, part).unflatten(-1, (-1, 2)).contiguous())
            out[..., 2 * chi:2 * chi + 2, :] = part.unflatten(-1, (2, 3))
        return out

    def dw(self, psi):
        return (4.0 - M0) * psi + self.hop(psi)

    def dfull(self, psi):
        return self.dw(self.along_s(self.W, psi)) + self.along_s(self.L1, psi)

    def g5(self, psi):
        out = psi.clone()
        out[..., 2:, :] *= -1
        return out

    def c(self, psi, p):
        psi = psi * self.mask[p]
        u = self.along_s(self.M5, self.hop(psi))
        return psi - self.along_s(self.M5, self.hop(u))

    def cdag(self, psi, p):
        psi = psi * self.mask[p]
        u = self.hop(self.along_s(self.M5, self.g5(psi), True))
        return psi - self.g5(self.hop(self.along_s(self.M5, u, True)))

    def solve_normal(self, b, p, batch=0, tol=2e-13, most=6000):
        """C C^dag x = b on parity p by conjugate gradient; the first `batch` dimensions of b
        are independent systems."""
        b = b * self.mask[p]
        dot = lambda v, w: torch.view_as_real(v.conj() * w)[..., 0].flatten(batch).sum(-1)  # noqa: E731
        wide = lambda a: a.reshape(a.shape + (1,) * (b.dim() - batch))  # noqa: E731
        x, r, p_ = torch.zeros_like(b), b.clone(), b.clone()
        rr = dot(r, r)
        stop = tol * tol * rr
        for it in range(most):
            q = self.cdag(p_, p)
            al = rr / dot(q, q)
            x += wide(al) * p_
            r -= wide(al) * self.c(q, p)
            new = dot(r, r)
            p_ = r + wide(new / rr) * p_
            rr = new
            if it % 16 == 0 and bool((rr <= stop).all()):
                break
        return x

    def solve_full(self, eta, p, batch=0):
        ep = self.along_s(self.S1, eta)
        eo = ep * self.mask[1 - p]
        b = ep * self.mask[p] - self.along_s(self.M5, self.hop(eo))
        phi = self.cdag(self.solve_normal(b, p, batch), p)
        phi = phi + eo - self.along_s(self.M5, self.hop(phi))
        return self.along_s(self.S2, phi)


def _reals(psi):
    return torch.view_as_real(psi.contiguous()).reshape(-1)


def exact(case, seed):
    dims, kind = _dims(case), case["kind"]
    U = _gauge(dims, case["eps"], seed)
    if kind == "ragged":
        return [_reals(_exact_solve(_Exact(dims, ns, mq, case["weights"], U), _source(dims, ns, seed, tag=2 + k), 1,
                                    False)) for k, (ns, mq) in enumerate(_masses(case))]
    ex = _Exact(dims, case["ns"], case["mq"], case["weights"], U)
    if kind == "prop":
        return _exact_prop(ex, case, seed)
    if kind == "solve":
        if inputs.volume(dims) * case["ns"] > 12 ** 3 * 24 * 8:
            return None  # the conjugate gradient in torch takes over 20 seconds
        on = case["parity"] if case["normal"] else None
        x = _exact_solve(ex, _source(dims, case["ns"], seed, parity=on), case["parity"], case["normal"])
        return _reals(x)
    psi, op, p = ex.field(_source(dims, case["ns"], seed)), case["op"], case["parity"]
    if op in ("DEO", "DOE"):
        q = 0 if op == "DEO" else 1
        out = ex.hop(psi * ex.mask[1 - q]) * ex.mask[q]
    elif op in ("M5", "M5T"):
        out = ex.along_s(ex.M5, psi * ex.mask[p], op == "M5T")
    elif op == "C":
        out = ex.c(psi, p)
    elif op == "CDAG":
        out = ex.cdag(psi, p)
    elif op == "CCDAG":
        out = ex.c(ex.cdag(psi, p), p)
    else:
        out = ex.dfull(psi) if op == "DFULL" else ex.dw(psi)
    return _reals(out)


def _exact_solve(ex, rhs, parity, normal):
    eta = ex.field(rhs)
    return ex.solve_normal(eta, parity) if normal else ex.solve_full(eta, parity)


def _exact_prop(ex, case, seed):
    """The 12 point sources on their chirality's wall slice; q = P- psi(0) + P+ psi(Ns-1)."""
    dims, ns = _dims(case), case["ns"]
    x0 = [int(v) for v in np.random.RandomState(int(seed) & 0x7FFFFFFF).randint(0, dims)]
    eta = torch.zeros((12, dims[3], dims[2], dims[1], dims[0], ns, 4, 3), dtype=torch.complex128, device="cuda")
    for k in range(12):
        spin, colour = divmod(k, 3)
        eta[k, x0[3], x0[2], x0[1], x0[0], 0 if spin < 2 else ns - 1, spin, colour] = 1.0
    psi = ex.solve_full(eta, 1, batch=1)
    q = torch.cat([psi[..., ns - 1, :2, :], psi[..., 0, 2:, :]], dim=-2)  # [12, t, z, y, x, spin, colour]
    return _reals(q.reshape(12, -1, 12).permute(1, 2, 0))
