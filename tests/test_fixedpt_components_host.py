"""The FP64 stencil's fixed-point hop sums (csrc/fixedpt.cuh), built for the host, where components of a site or of
its neighbours differ in size: what FP64 arithmetic keeps of the small ones is kept."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import synth
from oracle import gamma

HERE = os.path.dirname(os.path.abspath(__file__))
DIMS = (4, 6, 2, 8)
VOL = int(np.prod(DIMS))
KAPPA = 0.25  # 1 / (2 m_W + 8) at m_W = -2


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fx") / "fixedpt_check.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"),
                    os.path.join(HERE, "native", "fixedpt_check.cpp"), "-o", out], check=True)
    so = ctypes.CDLL(out)
    so.dslash_check.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_double, ctypes.c_double,
                                ctypes.c_int] + [ctypes.c_void_p] * 7
    return so


def _check(lib, u, psi, mu=0.3, g5=0):
    """Whether the field takes fixed point, D_W psi by it and by the FP64 hops, their distances from extended
    precision ([12][V][re, im]), and the sites that fixed point serves."""
    d = np.array(DIMS, np.int32)
    un = np.ascontiguousarray(u.reshape(4, VOL, 9).transpose(0, 2, 1))
    pn = np.ascontiguousarray(psi.reshape(VOL, 12).T)
    fx, f64, efx, ef64 = [np.zeros((12, VOL, 2)) for _ in range(4)]
    usable = np.zeros(VOL, np.int32)
    ok = lib.dslash_check(d.ctypes.data, -1, -2.0, mu, g5, un.ctypes.data, pn.ctypes.data, fx.ctypes.data,
                          f64.ctypes.data, efx.ctypes.data, ef64.ctypes.data, usable.ctypes.data)
    return bool(ok), fx, f64, efx, ef64, usable.astype(bool)


@pytest.mark.parametrize("g5", [0, 1])
@pytest.mark.parametrize("spins", [(0,), (1, 3), (2,)])
def test_negative_zeros_add_nothing(lib, g5, spins):
    """Minus a source that fills only some spins of a few sites: its other components are negative zeros, and a
    component whose neighbours are all zero stays exactly zero."""
    u, psi = synth.gauge_links(DIMS, 1), np.zeros((8, 2, 6, 4, 4, 3), complex)
    one = synth.gaussian_source(DIMS, 2)
    for site in ((0, 0, 0, 0), (3, 1, 4, 2), (7, 0, 5, 3)):
        for s in spins:
            psi[site][s] = one[site][s]
    psi = -psi
    assert np.signbit(psi.real[1, 1, 1, 1]).all() and np.signbit(psi.imag[1, 1, 1, 1]).all()
    ok, fx, f64, _, _, usable = _check(lib, u, psi, g5=g5)
    assert ok and usable.all()
    zero = f64 == 0
    assert 0.2 < zero.mean() < 1
    assert not fx[zero].any()


# ------------------------------------------------------------------ colours that decouple
@pytest.fixture(scope="module")
def field_usable(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fx") / "linkfield_check.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"),
                    os.path.join(HERE, "native", "linkfield_check.cpp"), "-o", out], check=True)
    so = ctypes.CDLL(out)
    so.field_usable.argtypes = [ctypes.c_void_p, ctypes.c_longlong]
    so.convert.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]

    def usable(u):
        u = np.ascontiguousarray(u)
        return bool(so.field_usable(u.ctypes.data, u.size // 9))

    so.large_spins.argtypes = [ctypes.c_void_p, ctypes.c_double] + [ctypes.c_void_p] * 3
    usable.lib = so
    return usable


def _blocks():
    """SU(2) links in colours 0 and 2."""
    rng = np.random.default_rng(5)
    a = rng.standard_normal((4, 8, 2, 6, 4, 4))
    a /= np.linalg.norm(a, axis=-1, keepdims=True)
    u = synth.unit_links(DIMS)
    p, q = a[..., 0] + 1j * a[..., 1], a[..., 2] + 1j * a[..., 3]
    u[..., 0, 0], u[..., 0, 2], u[..., 2, 0], u[..., 2, 2] = p, q, -q.conj(), p.conj()
    return u


def _phases():
    th = np.random.default_rng(6).uniform(-3, 3, (4, 8, 2, 6, 4, 3))
    u = synth.unit_links(DIMS)
    for c in range(3):
        u[..., c, c] = np.exp(1j * (th[..., c] - th.mean(-1)))
    return u


def _monomial():
    """Every link a permutation of the colours with phases: colours stay apart from site to site."""
    rng = np.random.default_rng(7)
    return np.stack([np.eye(3)[rng.permutation(3)] for _ in range(4 * VOL)]).reshape(_phases().shape) * _phases().sum(
        -1, keepdims=True) / abs(_phases().sum(-1, keepdims=True))


DECOUPLED = {"unit": lambda: synth.unit_links(DIMS), "phases": _phases, "su2 blocks": _blocks, "monomial": _monomial}


def _terms(u, psi, mu):
    """Per component, the sum of the moduli of D_W psi's terms, over re and im: [12][V]."""
    g = gamma.GAMMA
    a = np.abs(psi.real) + np.abs(psi.imag)
    out, au = a.copy(), np.abs(u.real) + np.abs(u.imag)
    for nu in range(4):
        ax = 3 - nu
        ef, eb = (np.exp(mu), np.exp(-mu)) if nu == 3 else (1.0, 1.0)
        p = np.abs(np.eye(4)) + np.abs(g[nu])
        out += KAPPA * ef * np.einsum("tzyxab,ij,tzyxjb->tzyxia", au[nu], p, np.roll(a, -1, ax))
        out += KAPPA * eb * np.roll(np.einsum("tzyxba,ij,tzyxjb->tzyxia", au[nu], p, a), 1, ax)
    return out.reshape(VOL, 12).T


@pytest.mark.parametrize("field", DECOUPLED)
@pytest.mark.parametrize("small", [1e-2, 1e-6, 1e-10, 1e-20])
def test_decoupled_colours(lib, field, small):
    """Fields whose links leave colours apart, a colour of the source smaller than the others: the field takes the
    FP64 hops, or every component is off by at most the FP64 chains' bound, sixteen roundings of its own terms
    (a projection, six multiply-adds, eight hops and the site itself)."""
    u, psi = DECOUPLED[field](), synth.gaussian_source(DIMS, 2)
    psi[..., 1] *= small
    ok, _, _, efx, _, usable = _check(lib, u, psi)
    bound = 2.0 ** -49 * _terms(u, psi, 0.3)[:, :, None]
    assert not ok or (efx <= bound)[:, usable].all()


@pytest.mark.parametrize("field", DECOUPLED)
def test_decoupled_fields_are_refused(field_usable, field):
    assert not field_usable(DECOUPLED[field]())


@pytest.mark.parametrize("eps", [0.1, 0.3, 0.5, 2.0])
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 4, 4, 4), (8, 8, 8, 8)])
def test_mixing_fields_are_accepted(field_usable, eps, dims):
    for seed in range(3):
        assert field_usable(synth.gauge_links(dims, seed, eps))
        assert field_usable(3.0 * synth.gauge_links(dims, seed, eps))


def test_where_the_field_rule_ends(field_usable):
    u = synth.gauge_links(DIMS, 1, 2.0)
    flat = u.reshape(-1, 3, 3)
    one = flat[100].copy()
    top = max(abs(one.real).max(), abs(one.imag).max())
    for small, want in ((2.0 ** -19, True), (2.0 ** -21, False), (0.0, False)):
        flat[100] = one
        flat[100][2, 0] = top * small * 1j
        assert field_usable(u) == want
    flat[100] = one
    n = len(flat)
    weak = synth.gauge_links(DIMS, 3, 1e-3).reshape(-1, 3, 3)  # off-diagonal entries about 1e-3
    for share, want in ((0.45, True), (0.55, False)):
        v = flat.copy()
        v[:int(share * n)] = weak[:int(share * n)]
        assert field_usable(v) == want
    assert not field_usable(synth.gauge_links(DIMS, 4, 1e-5))


# ------------------------------------------------------------------ spins
def _split_source(kind, small):
    """Sources whose neighbourhoods hold spins of very different size that a hop keeps apart."""
    psi = synth.gaussian_source(DIMS, 2)
    if kind == "spin":  # gamma_3 and gamma_4 join spins 0, 2 and 1, 3; the others 0, 3 and 1, 2
        psi[..., 1:, :] *= small
        psi[:, :, 1::2] *= 0
        psi[:, :, :, 1::2] *= 0
    if kind == "point":  # points of one spin beside points of another
        one = psi.copy()
        psi = np.zeros_like(psi)
        psi[2, 0, 1, 1, 0], psi[2, 0, 3, 1, 2] = one[0, 0, 0, 0, 0], one[0, 0, 1, 0, 2]
        psi[2, 0, 1, 3, 1] = small * one[1, 0, 0, 0, 1]
    return psi


def _spin_sizes(psi, mu):
    """Largest component of each spin over a site's neighbours, with the time hops' factors: [V][4]."""
    a = np.maximum(np.abs(psi.real), np.abs(psi.imag)).max(-1)
    m = np.zeros_like(a)
    for ax in range(4):
        for sh in (1, -1):
            m = np.maximum(m, np.roll(a, sh, ax) * (np.exp(-sh * mu) if ax == 0 else 1.0))
    return m.reshape(VOL, 4)


@pytest.mark.parametrize("mu", [0.0, 0.3, -5.0])
@pytest.mark.parametrize("small", [1e-3, 1e-10, 1e-20])
@pytest.mark.parametrize("kind", ["spin", "point"])
def test_sites_with_a_small_spin_are_refused(lib, kind, small, mu):
    """A site keeps fixed point only if each spin, over its neighbours, is zero or reaches 2^-6 of the largest (up
    to a factor of four: the mantissas' share of the words and the time hops' factors by their exponents). The
    other sites take the FP64 hops."""
    u, psi = synth.gauge_links(DIMS, 1), _split_source(kind, small)
    ok, fx, f64, efx, _, usable = _check(lib, u, psi, mu)
    assert ok
    m = _spin_sizes(psi, mu)
    top = m.max(1)[:, None]
    assert ((m == 0) | (m >= 2.0 ** -8 * top))[usable].all()
    assert usable[top[:, 0] == 0].all()
    assert usable[((m == 0) | (m >= 2.0 ** -4 * top)).all(1)].all()
    assert not usable.all()
    assert not fx[:, usable][f64[:, usable] == 0].any()


def test_real_links_are_refused(field_usable):
    """Real links join real and imaginary parts through the gammas alone, as single colours would be."""
    q, r = np.linalg.qr(np.random.default_rng(8).standard_normal((4, 8, 2, 6, 4, 3, 3)))
    u = (q * np.sign(np.diagonal(r, axis1=-2, axis2=-1))[..., None, :]).astype(complex)
    assert not field_usable(u) and not field_usable(1j * u)
    assert field_usable(u * np.exp(0.1j))


def test_gaussian_sources_are_served(lib):
    for seed in range(4):
        for mu in (0.0, 0.3, 1.4, -5.0, 16.0):
            assert _check(lib, synth.gauge_links(DIMS, seed, 0.5), synth.gaussian_source(DIMS, seed), mu)[5].all()


def test_subnormal_neighbours(lib):
    """A neighbourhood of subnormal components only is not zero."""
    psi = 1e-312 * synth.gaussian_source(DIMS, 2)
    assert not _check(lib, synth.gauge_links(DIMS, 1), psi)[5].any()


@pytest.mark.parametrize("uexp", [-8, -1, 0, 3, 8])
def test_link_components_round_to_nearest(field_usable, uexp):
    """The links' copy by shifts: x 2^(58 - uexp) to nearest, ties to even, over sizes from the scale to nothing."""
    rng = np.random.default_rng(9)
    x = rng.uniform(-1, 1, 20000) * 2.0 ** rng.integers(-70, 1, 20000)
    ties = (rng.integers(-2 ** 20, 2 ** 20, 4000) + 0.5) * 2.0 ** -58  # halfway between two units
    x = np.concatenate([x, ties, [0.0, -0.0, 1.0, -1.0, 1 - 2.0 ** -53, 2.0 ** -59, -2.0 ** -59, 2.0 ** -60, 3 * 2.0 ** -60]])
    x = np.ascontiguousarray(np.concatenate([x * 2.0 ** uexp, [5e-324, -5e-324, 1e-310]]))
    got, want = np.zeros(len(x), np.int64), np.zeros(len(x), np.int64)
    field_usable.lib.convert(x.ctypes.data, len(x), uexp, got.ctypes.data, want.ctypes.data)
    assert (got == want).all()


@pytest.mark.parametrize("mu", [0.0, 0.3, 1.3])
@pytest.mark.parametrize("spins", [(0,), (1,), (0, 1), (2, 3), (0, 2), (0, 1, 2)])
@pytest.mark.parametrize("small", [1e-2, 1e-5, 1e-9, 1e-20])
def test_small_components_where_fixed_point_is_kept(lib, spins, small, mu):
    """Whatever spins are small on whatever sites: where fixed point is kept, each spin's sum has terms of at least
    2^-9 of the largest neighbour component (fx_even: 2^-6 and a factor of four), and the sums meet their own bound,
    2^-49 of four times that component."""
    u, psi = synth.gauge_links(DIMS, 11), synth.gaussian_source(DIMS, 12)
    some = np.random.default_rng(13).random((8, 2, 6, 4)) < 0.7
    for s in spins:
        psi[..., s, :] *= np.where(some, small, 1.0)[..., None]
    ok, fx, f64, efx, _, usable = _check(lib, u, psi, mu)
    assert ok and usable.any()
    own = (np.abs(psi.real) + np.abs(psi.imag)).reshape(VOL, 12).T
    terms = (_terms(u, psi, mu) - own).reshape(4, 3, VOL).max(1)
    top = _spin_sizes(psi, mu).max(1)
    assert (terms >= 2.0 ** -9 * KAPPA * top)[:, usable].all()
    hop = 2.0 ** -49 * 4 * top * KAPPA * max(1.0, np.exp(abs(mu)))
    bound = hop[None, :, None] + 2.0 ** -53 * (3 * np.abs(fx) + 2 * own[:, :, None])
    assert (efx <= bound)[:, usable].all()


@pytest.mark.parametrize("mu", [0.0, 0.3, 1.3])
@pytest.mark.parametrize("spins", [(), (0,), (1,), (0, 1), (2, 3), (0, 2), (0, 1, 2)])
@pytest.mark.parametrize("small", [1e-2, 1e-20])
def test_large_sums_have_large_terms(field_usable, spins, small, mu):
    """fx_large: sums of at least 2^-3 of the largest neighbour component (2^-5 with the time hops' factors) have terms
    of 2^-9 of it, over at most three colours and both parts; nearly every sum of a Gaussian field is large, none of a
    spin without large terms."""
    u, psi = synth.gauge_links(DIMS, 11), synth.gaussian_source(DIMS, 12)
    psi[..., list(spins), :] *= small
    un = np.ascontiguousarray(u.reshape(4, VOL, 9).transpose(0, 2, 1))
    pn = np.ascontiguousarray(psi.reshape(VOL, 12).T)
    d, large = np.array(DIMS, np.int32), np.zeros((4, VOL), np.int32)
    field_usable.lib.large_spins(d.ctypes.data, mu, un.ctypes.data, pn.ctypes.data, large.ctypes.data)
    large = large.astype(bool)
    own = (np.abs(psi.real) + np.abs(psi.imag)).reshape(VOL, 12).T
    terms = (_terms(u, psi, mu) - own).reshape(4, 3, VOL).max(1)
    top = _spin_sizes(psi, mu).max(1)
    assert (terms >= 2.0 ** -9 * KAPPA * top)[large].all()
    assert not large[terms < 2.0 ** -9 * KAPPA * top].any()
    if not spins:
        assert large.mean() > 0.999
