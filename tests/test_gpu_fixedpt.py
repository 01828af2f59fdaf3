"""The fixed-point FP64 stencil and Lanczos step on the GPU, where their shapes and dispatch can go wrong.

Stencil: 1e-13 of the largest output (the FP64 bound of the other stencil tests) below, at and above the volume
where the four-thread shape ends, with half-filled chunks, scaled fields, fields and sites that take the
FP64 hops. Lanczos: integer sums inside a block and a fixed split of the sums over blocks, so
the results are the same bits for every pinned shape, evaluation interval and pass.
"""
import numpy as np
import pytest

import synth
from oracle import deflation, lanczos, wilson

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


def _close(got, ref):
    assert np.abs(got - ref).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 6, 2, 2), (16, 16, 8, 14), (16, 12, 10, 16)])
def test_stencil_shapes(ovl, ctx, dims):
    u, psi = synth.gauge_links(dims, 21), synth.gaussian_source(dims, 22, nrhs=3)
    lat = _lat(ovl, ctx, dims, u)
    got = _dw(ovl, lat, psi)
    for r in range(3):
        _close(got[r], wilson.apply_dw(u, psi[r], -2.0, 0.3, -1))
        assert np.array_equal(got[r], _dw(ovl, lat, psi[r]))  # alone as in a batch
    ovl.ovl_destroy_lattice(lat)


@pytest.mark.parametrize("dims", [(4, 4, 2, 6), (16, 12, 10, 16)])
@pytest.mark.parametrize("field", ["scaled", "zero link", "huge"])
def test_stencil_other_fields(ovl, ctx, dims, field):
    u, psi = synth.gauge_links(dims, 23).copy(), synth.gaussian_source(dims, 24)
    if field == "scaled":
        u *= 3.0
    if field == "huge":
        u *= 1e6
    if field == "zero link":
        u.reshape(-1, 3, 3)[77] = 0
    lat = _lat(ovl, ctx, dims, u)
    _close(_dw(ovl, lat, psi), wilson.apply_dw(u, psi, -2.0, 0.3, -1))
    ovl.ovl_set_links(lat, synth.gauge_links(dims, 25), ovl.OVL_F64)  # the handle takes the other route again
    _close(_dw(ovl, lat, psi), wilson.apply_dw(synth.gauge_links(dims, 25), psi, -2.0, 0.3, -1))
    ovl.ovl_destroy_lattice(lat)


@pytest.mark.parametrize("dims", [(4, 4, 2, 6), (16, 12, 10, 16)])
def test_stencil_special_values(ovl, ctx, dims):
    u, psi = synth.gauge_links(dims, 26), synth.gaussian_source(dims, 27)
    lat = _lat(ovl, ctx, dims, u)
    for mu in (20.0, 0.0):  # beyond the factors' range, and without factors
        _close(_dw(ovl, lat, psi, mu), wilson.apply_dw(u, psi, -2.0, mu, -1))
    _close(_dw(ovl, lat, 1e-300 * psi), wilson.apply_dw(u, 1e-300 * psi, -2.0, 0.3, -1))
    _close(_dw(ovl, lat, 1e300 * psi), wilson.apply_dw(u, 1e300 * psi, -2.0, 0.3, -1))
    assert not _dw(ovl, lat, 0 * psi).any()
    for value in (np.nan, np.inf):
        q = psi.copy()
        q[1, 1, 2, 3, 2, 1] = value
        with np.errstate(invalid="ignore"):
            ref = wilson.apply_dw(u, q, -2.0, 0.3, -1)
        got = _dw(ovl, lat, q)
        bad = ~np.isfinite(ref).all(axis=(-1, -2))
        assert bad.sum() >= 6
        assert (~np.isfinite(got).all(axis=(-1, -2)) == bad).all()
        _close(got[~bad], ref[~bad])
    ovl.ovl_destroy_lattice(lat)


def _solve(ovl, lat, b, variant, **kw):
    vol = b[0, ..., 0, 0].size
    ovl.ovl_set_pair_variant(vol, ovl.OVL_PREC_F64, variant)
    try:
        bt = torch.from_numpy(np.ascontiguousarray(b)).cuda()
        xt = torch.empty_like(bt)
        st, info = ovl.ovl_apply_sign(lat, ovl.ovl_sign_params_default(mu=0.3, **kw), bt, xt)
    finally:
        ovl.ovl_set_pair_variant(vol, ovl.OVL_PREC_F64, -1)
    assert st == ovl.OVL_OK
    return xt.cpu().numpy(), [ovl.ovl_get_tridiag(lat, r) for r in range(len(b))]


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 2, 6, 6), (10, 8, 6, 12), (14, 10, 10, 10), (10, 10, 10, 10)])
@pytest.mark.parametrize("two_pass", [0, 1])
def test_lanczos_same_bits(ovl, ctx, dims, two_pass):
    k = 24
    u, b = synth.gauge_links(dims, 31), synth.gaussian_source(dims, 32, nrhs=2)
    lat = _lat(ovl, ctx, dims, u)
    x0, t0 = _solve(ovl, lat, b, 0, fixed_k=k, check_every=24, two_pass=two_pass)
    for variant, every in ((1, 24), (0, 5), (1, 7)):
        x, t = _solve(ovl, lat, b, variant, fixed_k=k, check_every=every, two_pass=two_pass)
        assert np.array_equal(x, x0)
        for r in range(2):
            for p, q in zip(t[r], t0[r]):
                assert np.array_equal(p, q)
    x, t = _solve(ovl, lat, b[1:], 1, fixed_k=k, check_every=24, two_pass=two_pass)
    assert np.array_equal(x[0], x0[1])  # alone as in a batch
    ovl.ovl_destroy_lattice(lat)


@pytest.mark.parametrize("field", ["scaled", "zero link", "point source"])
def test_lanczos_other_fields(ovl, ctx, field):
    """A field with a scale of its own (fixed point), one without a common scale (FP64 vectors), and a source
    that is a negative zero but for one site, against Algorithm 4 at equal k: 1e-10, as the other
    equal-k comparisons."""
    dims, k = (4, 2, 6, 4), 20
    u, b = synth.gauge_links(dims, 33).copy(), synth.gaussian_source(dims, 34)
    if field == "scaled":
        u *= 1.5
    elif field == "point source":
        one = b[1, 2, 0, 3].copy()
        b = np.full_like(b, complex(-0.0, -0.0))
        b[1, 2, 0, 3] = one
    else:
        u.reshape(-1, 3, 3)[41] = 0
    lat = _lat(ovl, ctx, dims, u)
    x, t = _solve(ovl, lat, b[None], -1, fixed_k=k, check_every=6)
    a, ah = deflation.sparse_hw(u, dims, -2.0, 0.3), deflation.sparse_hw(u, dims, -2.0, -0.3)
    xo, sto = lanczos.direct_lanczos_lr(lambda v: (a @ v.ravel()).reshape(v.shape),
                                        lambda w: (ah @ w.ravel()).reshape(w.shape), b, k)
    for got, name in zip(t[0], ("alpha", "beta", "delta")):
        assert np.abs(got - sto[name]).max() < 1e-10 * np.abs(sto[name]).max()
    assert np.linalg.norm(x[0] - xo) < 1e-10 * np.linalg.norm(xo)
    ovl.ovl_destroy_lattice(lat)
