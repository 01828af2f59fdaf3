"""Performance cases: what a program asks of the library, through its public entry points.

Two families. "dw" cases are one application of D_W or H_W = gamma5 D_W (ovl_apply_DW): the
operator by itself, as an eigensolver or an outer solver calls it. "sign" cases are whole solves
x = sign(H_W(mu)) b (ovl_apply_sign) by the direct two-sided Lanczos method, by the multishift BiCG
with FP64 reliable updates and by restarted FOM.

Inputs follow the synthetic ensemble of `synth`: SU(3) links of spread eps = 0.5 and Gaussian
sources, made on the GPU from the seed; m_W = -2, antiperiodic time. Deflated solves need
eigenpairs, so their links are a gauge transform of constant diagonal SU(3) phases, whose eigenvectors are
known in closed form (plane waves); the library does the same work on them as on any other field.

Solves stop at the library's default tolerance 1e-10. They return x and the solve's status; the
numbers of steps and the timings in `info` are diagnostics.
"""
import math

import numpy as np
import torch

import paper_0910_1048_gb300 as ovl

M_W = -2.0
KAPPA = 1.0 / (2.0 * M_W + 8.0)
PREC = {"f64": ovl.OVL_PREC_F64, "f32": ovl.OVL_PREC_F32, "f16": ovl.OVL_PREC_F32_F16LINKS}
LINK_BYTES = {"f64": 4 * 144, "f32": 4 * 72, "f16": 4 * 24}  # per site


def _dw(name, lx, ly, lz, lt, fmt, nrhs=1, native=False, dagger=False, gamma5=True, mu=0.3):
    return {"name": name, "kind": "dw", "lx": lx, "ly": ly, "lz": lz, "lt": lt, "fmt": fmt, "nrhs": nrhs,
            "native": native, "dagger": dagger, "gamma5": gamma5, "mu": mu}


def _sign(name, lx, ly, lz, lt, method, mu=0.3, nrhs=1, defl=0, two_pass=False, s=0, k_max=3000):
    return {"name": name, "kind": "sign", "lx": lx, "ly": ly, "lz": lz, "lt": lt, "method": method, "mu": mu,
            "nrhs": nrhs, "defl": defl, "two_pass": two_pass, "s": s, "k_max": k_max}


def listed():
    return [
        # one operator call on the smallest lattice of the tests: launch latency
        _dw("dw_f64_4444", 4, 4, 4, 4, "f64"),
        # the matrix-vector product of an eigensolver on H_W(mu)^H (canonical layout, FP64)
        _dw("dw_f64_12_dagger", 12, 12, 12, 12, "f64", dagger=True),
        # FP64 residuals of a batch of systems (native layout), the solver's own layout
        _dw("dw_f64_16_batch8", 16, 16, 16, 16, "f64", nrhs=8, native=True, mu=0.2),
        # a large single-precision field in the library's layout
        _dw("dw_f32_32", 32, 32, 32, 32, "f32", native=True),
        # a batch of sources sharing the links
        _dw("dw_f32_24_batch16", 24, 24, 24, 24, "f32", nrhs=16, native=True),
        # 12-real FP16 links on a lattice of unequal extents, canonical layout, no gamma5
        _dw("dw_f16_ragged", 28, 20, 12, 30, "f16", gamma5=False, mu=0.1),
        # the smallest solve
        _sign("sign_direct_4444", 4, 4, 4, 4, "direct"),
        # 8^4 with 16 deflated eigenpairs
        _sign("sign_direct_8_defl16", 8, 8, 8, 8, "direct", mu=0.1, defl=16),
        # the benchmark's headline problem: 12^4, one source, FP64 two-sided Lanczos
        _sign("sign_direct_12", 12, 12, 12, 12, "direct"),
        # two sources, unequal extents, basis not stored (two passes)
        _sign("sign_direct_2pass_ragged", 14, 10, 12, 16, "direct", mu=0.2, nrhs=2, two_pass=True),
        # mixed precision: FP32 multishift iteration with FP64 reliable updates, 20 Zolotarev poles
        _sign("sign_mixed_16_batch4", 16, 16, 16, 16, "mixed", mu=0.2, nrhs=4, s=20, k_max=8000),
        # restarted FOM on A^2, FP64
        _sign("sign_fom_ragged", 8, 6, 6, 8, "fom", mu=0.3, s=20, k_max=40000),
    ]


def _extents(rng, lo, hi):
    """Even extents whose product is log-uniform in about [lo, hi]."""
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    while True:
        e = [2 * rng.randint(2, 18) for _ in range(4)]
        v = e[0] * e[1] * e[2] * e[3]
        if 0.8 * target <= v <= 1.25 * target and v <= hi:
            return e


def draw(rng):
    if rng.random() < 0.5:
        nrhs = rng.choice([1, 1, 1, 2, 3, 5, 8, 13, 16])
        e = _extents(rng, 256, min(1 << 20, (24 ** 4 * 16) // nrhs))
        c = _dw("", *e, rng.choice(["f64", "f64", "f32", "f32", "f16"]), nrhs=nrhs, native=rng.random() < 0.5,
                dagger=rng.random() < 0.3, gamma5=rng.random() < 0.7, mu=rng.choice([0.0, 0.1, 0.3, 0.5]))
    else:
        method = rng.choice(["direct", "direct", "direct", "mixed", "fom"])
        if method == "direct":
            defl = rng.choice([0, 0, 5, 16])
            two_pass = rng.random() < 0.3
            nrhs = rng.choice([1, 1, 2, 3])
            e = _extents(rng, 256, 20736 // nrhs)
            c = _sign("", *e, "direct", mu=rng.choice([0.0, 0.1, 0.2, 0.3]) if not defl else rng.choice([0.0, 0.1]),
                      nrhs=nrhs, defl=defl, two_pass=two_pass, k_max=6000)
        elif method == "mixed":
            nrhs = rng.choice([1, 2, 3, 4])
            e = _extents(rng, 256, min(65536, 131072 // nrhs))
            c = _sign("", *e, "mixed", mu=rng.choice([0.0, 0.2, 0.3]), nrhs=nrhs, s=rng.choice([16, 20]), k_max=8000)
        else:
            e = _extents(rng, 256, 2304)
            c = _sign("", *e, "fom", mu=rng.choice([0.0, 0.2, 0.3]), s=20, k_max=40000)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _cdot(a, b):
    return (a.conj() * b).sum(-1, keepdim=True)


def _su3(gen, shape, eps):
    """exp(i eps H), H traceless Hermitian as in `synth`: the Taylor series to rounding, its first two rows
    orthonormalised, the third their conjugate cross product."""
    g = torch.randn(shape + (3, 3, 2), dtype=torch.float64, device="cuda", generator=gen)
    g = torch.view_as_complex(g)
    one = torch.eye(3, dtype=g.dtype, device="cuda")
    h = 0.5 * eps * (g + g.conj().transpose(-1, -2))
    h = h - torch.diagonal(h, dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3 * one
    m = one + 0j * h
    for k in range(32, 0, -1):
        m = one + (1j / k) * (h[..., :, :, None] * m[..., None, :, :]).sum(-2)
    r0, r1 = m[..., 0, :], m[..., 1, :]
    r0 = r0 / _cdot(r0, r0).real.sqrt()
    r1 = r1 - _cdot(r0, r1) * r0
    r1 = r1 / _cdot(r1, r1).real.sqrt()
    r2 = torch.linalg.cross(r0, r1, dim=-1).conj()
    return torch.stack([r0, r1, r2], -2).contiguous()


def _dims(case):
    return case["lx"], case["ly"], case["lz"], case["lt"]


_AXIS = (-3, -4, -5, -6)  # site axis of direction x, y, z, t in a [..., t, z, y, x, 4, 3] spinor


def _phases(case, seed):
    """Constant diagonal phases theta[nu][colour] of a twisted field, their sum over colours zero."""
    r = np.random.default_rng(seed + 77)
    th = r.uniform(-0.25, 0.25, (4, 3))
    return th - th.mean(1, keepdims=True)


def _gauge(case, seed):
    """(U[4][Lt][Lz][Ly][Lx][3][3], G or None): links, and the gauge transform of a twisted field."""
    lx, ly, lz, lt = _dims(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000003 * seed + 17)
    if not case.get("defl"):
        return _su3(gen, (4, lt, lz, ly, lx), 0.5), None
    g = _su3(gen, (lt, lz, ly, lx), 2.0)
    th = torch.from_numpy(_phases(case, seed)).to("cuda")
    u = []
    for nu in range(4):
        gn = torch.roll(g, -1, dims=3 - nu)
        u.append(((g * torch.exp(1j * th[nu]))[..., :, None, :] * gn.conj()[..., None, :, :]).sum(-1))
    return torch.stack(u).contiguous(), g


def _source(case, seed, dtype=torch.complex128):
    lx, ly, lz, lt = _dims(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1000003 * seed + 9001)
    return torch.randn((case["nrhs"], lt, lz, ly, lx, 4, 3, 2), dtype=torch.float64, device="cuda",
                       generator=gen).view(torch.complex128).squeeze(-1).to(dtype).contiguous()


# Chiral gamma matrices of the library's operator (include/ovl.h): gamma_k = [[0, -i s_k], [i s_k, 0]],
# gamma_4 = [[0, 1], [1, 0]].
def _gammas():
    s = [np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]], complex)]
    z, one = np.zeros((2, 2)), np.eye(2)
    return [np.block([[z, -1j * a], [1j * a, z]]) for a in s] + [np.block([[z, one], [one, z]])]


_G5 = np.diag([1.0, 1.0, -1.0, -1.0])


def _momentum(case, seed):
    """Per FFT momentum and colour, H_W(p) = gamma5 D_W(p) of the twisted field: [t][z][y][x][3][4][4]."""
    lx, ly, lz, lt = _dims(case)
    th = _phases(case, seed)
    grid = np.meshgrid(*[2 * np.pi * np.fft.fftfreq(n) + (np.pi / lt if i == 0 else 0.0)
                         for i, n in enumerate((lt, lz, ly, lx))], indexing="ij")
    d = np.zeros((lt, lz, ly, lx, 3, 4, 4), complex) + np.eye(4)
    for nu, g in enumerate(_gammas()):
        f = np.exp(1j * (grid[3 - nu][..., None] + th[nu]))
        e = math.exp(case["mu"]) if nu == 3 else 1.0
        d -= KAPPA * (e * f[..., None, None] * (np.eye(4) - g) + (1 / e / f)[..., None, None] * (np.eye(4) + g))
    return _G5 @ d


def _twist(case):
    """exp(i pi t / Lt): turns antiperiodic time into periodic time."""
    return np.exp(1j * np.pi * np.arange(case["lt"]) / case["lt"]).reshape(-1, 1, 1, 1, 1, 1)


def _eigenpairs(case, seed, g):
    """The `defl` eigenpairs of H_W smallest in modulus: lam[m], R[m][...], L[m][...] with L^H R = 1."""
    lx, ly, lz, lt = _dims(case)
    h = _momentum(case, seed)
    w, v = np.linalg.eig(h)
    li = np.conj(np.swapaxes(np.linalg.inv(v), -1, -2))  # left eigenvectors in columns
    m = case["defl"]
    # whole degenerate pairs in a fixed order: by modulus, then by position
    order = np.lexsort((np.arange(w.size), np.round(np.abs(w.ravel()), 9)))[:m]
    t, z, y, x, c, k = np.unravel_index(order, w.shape)
    ar = [np.arange(n) for n in (lt, lz, ly, lx)]
    R = np.zeros((m, lt, lz, ly, lx, 4, 3), complex)
    L = np.zeros_like(R)
    for i in range(m):
        ph = np.exp(2j * np.pi * (ar[0].reshape(-1, 1, 1, 1) * t[i] / lt + ar[1].reshape(-1, 1, 1) * z[i] / lz
                                  + ar[2].reshape(-1, 1) * y[i] / ly + ar[3] * x[i] / lx)) / math.sqrt(lx * ly * lz * lt)
        ph = ph * _twist(case)[..., 0, 0]
        R[i, ..., c[i]] = ph[..., None] * v[t[i], z[i], y[i], x[i], c[i], :, k[i]]
        L[i, ..., c[i]] = ph[..., None] * li[t[i], z[i], y[i], x[i], c[i], :, k[i]]
    R, L = (torch.einsum("tzyxab,mtzyxsb->mtzyxsa", g, torch.from_numpy(a).to("cuda")).contiguous() for a in (R, L))
    return torch.from_numpy(w.ravel()[order].copy()).to("cuda"), R, L


class _State:
    """A lattice handle with its links, the inputs and the output buffer."""

    ctx = None

    def __init__(self, case, links, formats):
        if _State.ctx is None:
            _State.ctx = ovl.ovl_ctx_create(0)
        self.case = case
        self.lat = ovl.ovl_create_lattice(_State.ctx, _dims(case), -1)
        torch.cuda.synchronize()  # the library reads the links on a stream of its own
        ovl.ovl_set_links(self.lat, links, formats)

    def __del__(self):
        if getattr(self, "lat", None) is not None:
            ovl.ovl_destroy_lattice(self.lat)


def _flags(case):
    return ((ovl.OVL_DAGGER if case["dagger"] else 0) | (ovl.OVL_GAMMA5 if case["gamma5"] else 0)
            | (ovl.OVL_NATIVE if case["native"] else 0)
            | {"f64": 0, "f32": ovl.OVL_LINKS_F32, "f16": ovl.OVL_LINKS_F16R12}[case["fmt"]])


def prepare(case, seed):
    links, g = _gauge(case, seed)
    if case["kind"] == "dw":
        st = _State(case, links, {"f64": ovl.OVL_F64, "f32": ovl.OVL_F32, "f16": ovl.OVL_F16R12}[case["fmt"]])
        b = _source(case, seed, torch.complex128 if case["fmt"] == "f64" else torch.complex64)
        if case["native"]:
            st.b = torch.empty_like(b)
            ovl.ovl_to_native(st.lat, b, st.b)
        else:
            st.b = b
        st.x = torch.empty_like(st.b)
        st.flags = _flags(case)
        return st
    st = _State(case, links, ovl.OVL_F64 | ovl.OVL_F32)
    if case["defl"]:
        lam, R, L = _eigenpairs(case, seed, g)
        torch.cuda.synchronize()
        ovl.ovl_set_deflation(st.lat, M_W, case["mu"], R, L, lam)
    st.b = _source(case, seed)
    st.x = torch.empty_like(st.b)
    kw = {"direct": dict(method=ovl.OVL_DIRECT_2SL, precision=ovl.OVL_PREC_F64, check_every=25),
          "mixed": dict(method=ovl.OVL_MULTISHIFT_BICG, precision=ovl.OVL_PREC_F32),
          "fom": dict(method=ovl.OVL_FOM_RESTARTED, precision=ovl.OVL_PREC_F64)}[case["method"]]
    if case["s"]:
        kw.update(rational_kind=ovl.OVL_RAT_ZOLOTAREV, s=case["s"], spec_lo=0.03, spec_hi=2.75)
    st.p = ovl.ovl_sign_params_default(m_W=M_W, mu=case["mu"], tol=1e-10, k_max=case["k_max"],
                                       use_deflation=1 if case["defl"] else 0,
                                       two_pass=1 if case["two_pass"] else 0, **kw)
    return st


def run(st):
    if st.case["kind"] == "dw":
        ovl.ovl_apply_DW(st.lat, M_W, st.case["mu"], st.flags, st.b, st.x)
        return {"x": st.x}
    status, _ = ovl.ovl_apply_sign(st.lat, st.p, st.b, st.x)
    return {"x": st.x, "status": int(status)}


# Krylov steps (direct), BiCG iterations and Arnoldi steps a solve to 1e-10 of these sizes takes at least, and
# the arithmetic of one: stencils of 1368 flops a site and the recurrence's vector updates.
_STEPS = {"direct": 800, "mixed": 500, "fom": 500}
_STEP_FLOPS = {"direct": 2 * 1368 + 12 * 48, "mixed": 4 * 1368 + 12 * 64, "fom": 2 * 1368 + 12 * 16 * 20}


def work(case):
    vol = case["lx"] * case["ly"] * case["lz"] * case["lt"]
    nrhs = case["nrhs"]
    if case["kind"] == "dw":
        elt = 16 if case["fmt"] == "f64" else 8
        return {"bytes": vol * (LINK_BYTES[case["fmt"]] + nrhs * 2 * 12 * elt), "flops": 1368 * vol * nrhs}
    steps = _STEPS[case["method"]] if not case["defl"] else 150
    return {"bytes": vol * (LINK_BYTES["f64"] + (nrhs * 2 + case["defl"] * 2) * 12 * 16),
            "flops": steps * nrhs * vol * _STEP_FLOPS[case["method"]]}


# ------------------------------------------------------------------ the same in plain torch, 64 bits
def _plain_hops(u, psi, mu, dagger, gamma5):
    """D_W(mu) psi (or its adjoint, gamma5 after it) for psi[nrhs][t][z][y][x][4][3]."""
    g = [torch.from_numpy(a).to(psi) for a in _gammas()]
    g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=psi.dtype, device=psi.device)[:, None]
    one = torch.eye(4, dtype=psi.dtype, device=psi.device)
    out = psi.clone()
    for nu in range(4):
        ax = _AXIS[nu]
        ef, eb = (math.exp(mu), math.exp(-mu)) if nu == 3 else (1.0, 1.0)
        pf = torch.roll(psi, -1, dims=ax)
        pb = torch.roll((u[nu].conj().transpose(-1, -2)[..., None, :, :] * psi[..., None, :]).sum(-1), 1, dims=ax)
        pf = (u[nu][..., None, :, :] * pf[..., None, :]).sum(-1)
        if nu == 3:
            pf[:, -1] *= -1
            pb[:, 0] *= -1
        sg = -1.0 if dagger else 1.0  # D^H: gamma -> -gamma at -mu and the hops' factors exchanged
        if dagger:
            ef, eb = eb, ef
        out -= KAPPA * (ef * ((one - sg * g[nu])[:, :, None] * pf[..., None, :, :]).sum(-2)
                        + eb * ((one + sg * g[nu])[:, :, None] * pb[..., None, :, :]).sum(-2))
    return g5 * out if gamma5 else out


def _stored_links(u, fmt):
    if fmt == "f64":
        return u
    if fmt == "f32":
        return u.to(torch.complex64).to(torch.complex128)
    r = torch.view_as_real(u[..., :2, :]).to(torch.float32).to(torch.float16).to(torch.float64)
    r = torch.view_as_complex(r.contiguous())
    return torch.cat([r, torch.linalg.cross(r[..., 0, :], r[..., 1, :], dim=-1).conj()[..., None, :]], -2)


def exact(case, seed):
    vol = case["lx"] * case["ly"] * case["lz"] * case["lt"]
    links, g = _gauge(case, seed)
    if case["kind"] == "dw":
        b = _source(case, seed, torch.complex128 if case["fmt"] == "f64" else torch.complex64).to(torch.complex128)
        u = _stored_links(links, case["fmt"])
        out = torch.empty_like(b)
        for r in range(case["nrhs"]):
            out[r:r + 1] = _plain_hops(u, b[r:r + 1], case["mu"], case["dagger"], case["gamma5"])
        if case["native"]:
            out = out.reshape(case["nrhs"], vol, 12).transpose(1, 2).contiguous().reshape(out.shape)
        return {"x": out}
    b = _source(case, seed)
    if case["defl"]:
        # sign(H_W(p)) momentum by momentum: H_W(p)^2 = (a^2 + s.s) 1, so sign = H_W(p) / sqrt(H_W(p)^2)
        h = _momentum(case, seed)
        sq = (h @ h)[..., 0, 0]
        sgn = h / np.sqrt(sq)[..., None, None]
        chi = torch.einsum("tzyxab,ntzyxsa->ntzyxsb", g.conj(), b).cpu().numpy() / _twist(case)
        f = np.fft.fftn(chi, axes=(1, 2, 3, 4))
        f = np.einsum("tzyxcij,ntzyxjc->ntzyxic", sgn, f)
        chi = np.fft.ifftn(f, axes=(1, 2, 3, 4)) * _twist(case)
        return {"x": torch.einsum("tzyxab,ntzyxsb->ntzyxsa", g, torch.from_numpy(chi).to("cuda")).contiguous(),
                "status": None}
    if case["method"] != "direct" or vol > 256:
        return None
    # dense H_W and the Newton iteration for its sign, scaled by the determinant's modulus
    n = 12 * vol
    eye = torch.eye(n, dtype=torch.complex128, device="cuda").reshape((n,) + tuple(b.shape[1:]))
    a = torch.cat([_plain_hops(links, e, case["mu"], False, True).reshape(-1, n) for e in eye.split(256)]).t()
    for it in range(60):
        inv = torch.linalg.inv(a)
        c = math.sqrt(float(torch.linalg.matrix_norm(inv) / torch.linalg.matrix_norm(a))) if it < 20 else 1.0
        new = 0.5 * (c * a + inv / c)
        done = float(torch.linalg.matrix_norm(new - a) / torch.linalg.matrix_norm(new)) < 1e-14
        a = new
        if done:
            break
    return {"x": (a @ b.reshape(-1, n).t()).t().reshape(b.shape).contiguous(), "status": None}
