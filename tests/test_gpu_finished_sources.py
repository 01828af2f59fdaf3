"""Sources of a batch that end early (retired, nothing to solve, broken down) take no part in the later steps of the
FP64 direct method, and leave the others' results as they are alone."""
import numpy as np
import pytest

import synth

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


def _solve(ovl, lat, b, **kw):
    bt = torch.from_numpy(np.ascontiguousarray(b)).cuda()
    xt = torch.empty_like(bt)
    st, info = ovl.ovl_apply_sign(lat, ovl.ovl_sign_params_default(mu=0.3, **kw), bt, xt)
    return st, info, xt.cpu().numpy()


def test_ended_sources_cost_no_step(ovl, ctx):
    """12^4, one source alone and beside seven that are zero: the step takes less than three sources' time."""
    dims = (12, 12, 12, 12)
    lat = ovl.ovl_create_lattice(ctx, dims, -1)
    ovl.ovl_set_links(lat, synth.gauge_links(dims, 0), ovl.OVL_F64)
    b = np.zeros((8,) + dims[::-1] + (4, 3), complex)
    b[3] = synth.gaussian_source(dims, 51)
    t = {}
    for name, src in (("alone", b[3:4]), ("batch", b)):
        for _ in range(2):
            st, info, x = _solve(ovl, lat, src, fixed_k=200, check_every=20)
            assert st == ovl.OVL_OK
        t[name] = info[0]["t_kernel_ms"], info[0]["t_update_ms"]
        if name == "alone":
            alone = x[0]
    ovl.ovl_destroy_lattice(lat)
    assert np.array_equal(x[3], alone)
    assert t["batch"][0] < 3 * t["alone"][0] and t["batch"][1] < 3 * t["alone"][1], t


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (8, 8, 8, 10)])
@pytest.mark.parametrize("two_pass", [0, 1])
def test_batch_of_sources_that_end(ovl, ctx, dims, two_pass):
    """A source that breaks down at the start, a zero one and two Gaussian ones that converge at their own steps: the
    same results as alone, bit for bit."""
    n = 12 * int(np.prod(dims))
    rng = np.random.default_rng(52)
    e, _ = np.linalg.qr(rng.standard_normal((n, 3)) + 1j * rng.standard_normal((n, 3)))
    lat = ovl.ovl_create_lattice(ctx, dims, -1)
    ovl.ovl_set_links(lat, synth.gauge_links(dims, 53), ovl.OVL_F64)
    # r~ = b - L R^H b is orthogonal to r = b - R L^H b for b = e0 + e1 + e2
    ovl.ovl_set_deflation(lat, -2.0, 0.3, e[:, 0][None], (e[:, 0] + 2.0 * e[:, 2])[None], np.array([0.7 + 0.1j]))
    shape = dims[::-1] + (4, 3)
    b = np.stack([(e[:, 0] + e[:, 1] + e[:, 2]).reshape(shape), np.zeros(shape, complex),
                  synth.gaussian_source(dims, 54), synth.gaussian_source(dims, 55)])
    kw = dict(tol=1e-3, k_max=300, check_every=10, use_deflation=1, two_pass=two_pass)
    st, info, x = _solve(ovl, lat, b, **kw)
    assert info[0]["status"] == ovl.OVL_EBREAKDOWN and info[0]["iterations"] == 0
    assert info[1]["status"] == ovl.OVL_OK and info[1]["iterations"] == 0 and not x[1].any()
    for r in range(4):
        _, one, xr = _solve(ovl, lat, b[r:r + 1], **kw)
        assert one[0]["status"] == info[r]["status"] and one[0]["iterations"] == info[r]["iterations"]
        assert np.array_equal(xr[0], x[r]), r
    ovl.ovl_destroy_lattice(lat)
