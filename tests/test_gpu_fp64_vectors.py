"""The FP64 direct method on FP64 vectors (fields that do not fit fixed point): every pair-stencil shape, the deferred
step, graphs and the allocation-free entry point, which fields that do fit never reach. The field is the seeded
ensemble with one zero link (no common scale); the operator and its oracles take any links."""
import numpy as np
import pytest

import synth
from oracle import krylov, lanczos, matsign, rational, wilson

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


def _links(dims, seed, eps=0.5):
    u = synth.gauge_links(dims, seed, eps).copy()
    u.reshape(-1, 3, 3)[7] = 0
    return u


def _lat(ovl, ctx, dims, u):
    lat = ovl.ovl_create_lattice(ctx, dims, -1)
    ovl.ovl_set_links(lat, u, ovl.OVL_F64)
    return lat


def _solve(ovl, lat, b, **kw):
    bt = torch.from_numpy(np.ascontiguousarray(b)).cuda()
    xt = torch.empty_like(bt)
    st, info = ovl.ovl_apply_sign(lat, ovl.ovl_sign_params_default(**kw), bt, xt)
    return st, info, xt.cpu().numpy()


def _rel(x, y):
    return np.linalg.norm(x - y) / np.linalg.norm(y)


def test_every_pair_shape_equal_k(ovl, ctx):
    dims, k = (12, 12, 12, 12), 24
    vol, u, b = 12 ** 4, _links(dims, 0), synth.gaussian_source(dims, 1000)
    lat = _lat(ovl, ctx, dims, u)
    xo, _, _ = krylov.direct_lanczos(u, dims, -2.0, 0.3, b, k)
    xs = []
    try:
        for var in range(9):
            ovl.ovl_set_pair_variant(vol, ovl.OVL_PREC_F64, var)
            st, info, x = _solve(ovl, lat, b, mu=0.3, fixed_k=k, check_every=8)
            assert st == ovl.OVL_OK and info[0]["iterations"] == k
            assert _rel(x, xo) < 1e-10, var
            xs.append(x)
    finally:
        ovl.ovl_set_pair_variant(vol, ovl.OVL_PREC_F64, -1)
        ovl.ovl_destroy_lattice(lat)
    for x in xs[1:]:  # the shapes differ only in the order of alpha's partial sums
        assert _rel(x, xs[0]) < 1e-12
    assert any(not np.array_equal(x, xs[0]) for x in xs[1:])  # (the fixed-point shapes give the same bits)


def test_shape_change_between_solves(ovl, ctx):
    dims = (2, 2, 2, 4)
    u, b = _links(dims, 35, 0.1), synth.gaussian_source(dims, 36)
    xs = matsign.sign_eig(wilson.dense_hw(u, dims, -2.0, 0.3), b.ravel()).reshape(b.shape)
    lat = _lat(ovl, ctx, dims, u)
    try:
        for var in (4, 7, 5, 7, 3):
            ovl.ovl_set_pair_variant(32, ovl.OVL_PREC_F64, var)
            st, info, x = _solve(ovl, lat, b, mu=0.3, tol=1e-10, k_max=384, check_every=16)
            assert st == ovl.OVL_OK, (var, info)
            assert _rel(x, xs) < 1e-10, var
    finally:
        ovl.ovl_set_pair_variant(32, ovl.OVL_PREC_F64, -1)
        ovl.ovl_destroy_lattice(lat)


@pytest.mark.parametrize("var", [7, 3])
def test_graph_chunks_equal_direct_launches(ovl, ctx, var):
    dims = (8, 8, 8, 8)
    u, b = _links(dims, 3), synth.gaussian_source(dims, 4, nrhs=2)
    lat = _lat(ovl, ctx, dims, u)
    xs = []
    try:
        ovl.ovl_set_pair_variant(8 ** 4, ovl.OVL_PREC_F64, var)
        for graphs in (1, 0):
            st, info, x = _solve(ovl, lat, b, mu=0.3, fixed_k=75, check_every=20, use_graphs=graphs)
            assert st == ovl.OVL_OK and all(i["iterations"] == 75 for i in info)
            xs.append(x)
        st, info, x = _solve(ovl, lat, b, mu=0.3, fixed_k=75, check_every=20, two_pass=1)
        assert st == ovl.OVL_OK and _rel(x, xs[0]) < 1e-12
    finally:
        ovl.ovl_set_pair_variant(8 ** 4, ovl.OVL_PREC_F64, -1)
        ovl.ovl_destroy_lattice(lat)
    assert np.array_equal(xs[0], xs[1])
    xo, _, _ = krylov.direct_lanczos(u, dims, -2.0, 0.3, b[0], 75)
    assert _rel(xs[0][0], xo) < 1e-10


@pytest.mark.parametrize("var", [7, 1])
def test_without_allocation(ovl, ctx, var):
    dims = (4, 4, 4, 4)
    u, b = _links(dims, 0), torch.from_numpy(synth.gaussian_source(dims, 1000, nrhs=2)).cuda()
    lat = _lat(ovl, ctx, dims, u)
    p = ovl.ovl_sign_params_default(mu=0.2, fixed_k=120)
    ovl.ovl_set_pair_variant(256, ovl.OVL_PREC_F64, var)
    try:
        x_ref, x = torch.empty_like(b), torch.full_like(b, float("nan"))
        assert ovl.ovl_apply_sign(lat, p, b, x_ref)[0] == ovl.OVL_OK
        assert ovl.ovl_apply_sign_noalloc(lat, p, b, x)[0] == ovl.OVL_OK
    finally:
        ovl.ovl_set_pair_variant(256, ovl.OVL_PREC_F64, -1)
        ovl.ovl_destroy_lattice(lat)
    assert float(torch.linalg.vector_norm(x - x_ref) / torch.linalg.vector_norm(x_ref)) < 1e-10


@pytest.mark.parametrize("var", [0, 1])
def test_multishift(ovl, ctx, var):
    """FP64 multishift (one and eight threads per site) against the dense g(A) b of the same rational function, with a
    field that does fit in between (the cached graphs follow the field)."""
    dims, eps = (2, 2, 2, 4), 1e-10
    u, b = _links(dims, 35, 0.1), synth.gaussian_source(dims, 36, nrhs=2)
    fit = synth.gauge_links(dims, 37, 0.3)
    lat = ovl.ovl_create_lattice(ctx, dims, -1)
    ovl.ovl_set_pair_variant(32, ovl.OVL_PREC_F64, var)
    try:
        for links in (u, fit, u):
            h = wilson.dense_hw(links, dims, -2.0, 0.3)
            ev = np.linalg.eigvals(h)
            lo, hi = 0.9 * float(np.abs(ev).min()), 1.1 * float(np.abs(ev).max())
            s, c, w, sg = rational.neuberger_for_spectrum(lo, hi, eps)
            ovl.ovl_set_links(lat, links, ovl.OVL_F64)
            st, info, x = _solve(ovl, lat, b, method=ovl.OVL_MULTISHIFT_BICG, mu=0.3, tol=eps, k_max=2000, spec_lo=lo,
                                 spec_hi=hi, check_every=10)
            assert st == ovl.OVL_OK and info[0]["poles"] == s
            for r in range(2):
                assert _rel(x[r].ravel(), lanczos.rational_sign_dense(h, b[r].ravel(), w, sg)) < 2e-9, r
    finally:
        ovl.ovl_set_pair_variant(32, ovl.OVL_PREC_F64, -1)
        ovl.ovl_destroy_lattice(lat)
