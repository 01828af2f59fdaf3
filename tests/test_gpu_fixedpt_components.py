"""FP64 operators and solves on the GPU where components differ in size: small components keep FP64's own accuracy.

D_W: sixteen roundings of a component's own terms (a projection, six multiply-adds, eight hops and the site), once for
the library and once for the oracle's FP64 sums: 2^-48 of the sum of the terms' moduli. Direct method: Algorithm 4 at
equal k to 1e-10 per colour, as the other equal-k comparisons."""
import numpy as np
import pytest

import synth
from oracle import deflation, gamma, lanczos, wilson

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ovl():
    import paper_0910_1048_gb300 as m
    return m


@pytest.fixture(scope="module")
def ctx(ovl):
    c = ovl.ovl_ctx_create(0)
    yield c
    ovl.ovl_ctx_destroy(c)


def _lat(ovl, ctx, dims, u):
    lat = ovl.ovl_create_lattice(ctx, dims, -1)
    ovl.ovl_set_links(lat, u, ovl.OVL_F64)
    return lat


def _dw(ovl, lat, psi, mu=0.3):
    inp = torch.from_numpy(np.ascontiguousarray(psi)).cuda()
    out = torch.empty_like(inp)
    ovl.ovl_apply_DW(lat, -2.0, mu, 0, inp, out)
    return out.cpu().numpy()


def _terms(u, psi, mu=0.3, kappa=0.25):
    a, au = np.abs(psi.real) + np.abs(psi.imag), np.abs(u.real) + np.abs(u.imag)
    out = a.copy()
    for nu in range(4):
        ax = 3 - nu
        ef, eb = (np.exp(mu), np.exp(-mu)) if nu == 3 else (1.0, 1.0)
        p = np.eye(4) + np.abs(gamma.GAMMA[nu])
        out += kappa * ef * np.einsum("tzyxab,ij,tzyxjb->tzyxia", au[nu], p, np.roll(a, -1, ax))
        out += kappa * eb * np.roll(np.einsum("tzyxba,ij,tzyxjb->tzyxia", au[nu], p, a), 1, ax)
    return out


def _close(got, u, psi):
    ref, bound = wilson.apply_dw(u, psi, -2.0, 0.3, -1), 2.0 ** -48 * _terms(u, psi)
    assert (np.abs(got.real - ref.real) <= bound).all() and (np.abs(got.imag - ref.imag) <= bound).all()


def _blocks(dims, seed):
    """SU(2) links in colours 0 and 2."""
    u = synth.unit_links(dims)
    a = np.random.default_rng(seed).standard_normal(u.shape[:5] + (4,))
    a /= np.linalg.norm(a, axis=-1, keepdims=True)
    p, q = a[..., 0] + 1j * a[..., 1], a[..., 2] + 1j * a[..., 3]
    u[..., 0, 0], u[..., 0, 2], u[..., 2, 0], u[..., 2, 2] = p, q, -q.conj(), p.conj()
    return u


@pytest.mark.parametrize("dims", [(4, 4, 2, 6), (16, 12, 10, 16)])
@pytest.mark.parametrize("field", ["unit", "su2 blocks"])
def test_stencil_of_decoupled_colours(ovl, ctx, dims, field):
    u = synth.unit_links(dims) if field == "unit" else _blocks(dims, 3)
    lat = _lat(ovl, ctx, dims, u)
    for small in (1.0, 1e-6, 1e-20):
        psi = synth.gaussian_source(dims, 41)
        psi[..., 1] *= small
        _close(_dw(ovl, lat, psi), u, psi)
    u2 = synth.gauge_links(dims, 25)  # the handle takes the other route again
    ovl.ovl_set_links(lat, u2, ovl.OVL_F64)
    _close(_dw(ovl, lat, psi), u2, psi)
    ovl.ovl_destroy_lattice(lat)


@pytest.mark.parametrize("two_pass", [0, 1])
def test_direct_solve_of_decoupled_colours(ovl, ctx, two_pass):
    dims, k = (4, 2, 6, 4), 20
    u, b = _blocks(dims, 4), synth.gaussian_source(dims, 42)
    b[..., 1] *= 1e-12
    lat = _lat(ovl, ctx, dims, u)
    bt = torch.from_numpy(b).cuda()
    xt = torch.empty_like(bt)
    st, _ = ovl.ovl_apply_sign(lat, ovl.ovl_sign_params_default(mu=0.3, fixed_k=k, check_every=6, two_pass=two_pass), bt, xt)
    assert st == ovl.OVL_OK
    x = xt.cpu().numpy()
    ovl.ovl_destroy_lattice(lat)
    a, ah = deflation.sparse_hw(u, dims, -2.0, 0.3), deflation.sparse_hw(u, dims, -2.0, -0.3)
    xo, _ = lanczos.direct_lanczos_lr(lambda v: (a @ v.ravel()).reshape(v.shape),
                                      lambda w: (ah @ w.ravel()).reshape(w.shape), b, k)
    for c in range(3):
        assert np.linalg.norm(x[..., c] - xo[..., c]) < 1e-10 * np.linalg.norm(xo[..., c])


@pytest.mark.parametrize("dims", [(4, 4, 2, 6), (16, 12, 10, 16)])
def test_negative_zeros_add_nothing(ovl, ctx, dims):
    """Minus a source with one spin at one site: components without a nonzero neighbour component are zero."""
    u, b = synth.gauge_links(dims, 43), np.zeros(dims[::-1] + (4, 3), complex)
    b[1, 0, 2, 1, 2] = synth.gaussian_source(dims, 44)[1, 0, 2, 1, 2]
    lat = _lat(ovl, ctx, dims, u)
    got, ref = _dw(ovl, lat, -b), wilson.apply_dw(u, -b, -2.0, 0.3, -1)
    ovl.ovl_destroy_lattice(lat)
    assert not got[ref == 0].any() and got.any()


@pytest.mark.parametrize("dims", [(4, 4, 2, 6), (16, 12, 10, 16)])
@pytest.mark.parametrize("small", [1e-6, 1e-20])
def test_stencil_of_small_spins(ovl, ctx, dims, small):
    """Spins far below the first at every site, on links that mix the colours; and such spins on half of the sites
    beside an ordinary field."""
    u, one = synth.gauge_links(dims, 45), synth.gaussian_source(dims, 46)
    lat = _lat(ovl, ctx, dims, u)
    spins, half = one.copy(), one.copy()
    spins[..., 1:, :] *= small
    half[::2, ..., 1:, :] *= small
    _close(_dw(ovl, lat, spins), u, spins)
    got, ref = _dw(ovl, lat, half), wilson.apply_dw(u, half, -2.0, 0.3, -1)
    assert np.abs(got - ref).max() <= 1e-13 * np.abs(ref).max()
    ovl.ovl_destroy_lattice(lat)


@pytest.mark.parametrize("small", [1e-6, 1e-14])
def test_direct_solve_of_a_source_with_small_spins(ovl, ctx, small):
    """On links that mix the colours the solve fills the small spins from the large one: each spin of x as Algorithm 4
    gives it at equal k, to 1e-10."""
    dims, k = (4, 2, 6, 4), 20
    u, b = synth.gauge_links(dims, 47), synth.gaussian_source(dims, 48)
    b[..., 1:, :] *= small
    lat = _lat(ovl, ctx, dims, u)
    bt = torch.from_numpy(b).cuda()
    xt = torch.empty_like(bt)
    assert ovl.ovl_apply_sign(lat, ovl.ovl_sign_params_default(mu=0.3, fixed_k=k, check_every=6), bt, xt)[0] == ovl.OVL_OK
    x = xt.cpu().numpy()
    ovl.ovl_destroy_lattice(lat)
    a, ah = deflation.sparse_hw(u, dims, -2.0, 0.3), deflation.sparse_hw(u, dims, -2.0, -0.3)
    xo, _ = lanczos.direct_lanczos_lr(lambda v: (a @ v.ravel()).reshape(v.shape),
                                      lambda w: (ah @ w.ravel()).reshape(w.shape), b, k)
    for s in range(4):
        assert np.linalg.norm(x[..., s, :] - xo[..., s, :]) < 1e-10 * np.linalg.norm(xo[..., s, :])
