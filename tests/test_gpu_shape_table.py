"""The pair-shape table: the FP64 direct method's fixed-point step and its step on FP64 vectors are different kernels
with shapes of their own, tuned apart, whichever runs first."""
import ctypes

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FP64_VECTORS, FIXED_POINT = 0, 3  # keys of the library's table


@pytest.fixture(scope="module")
def ovl():
    import paper_0910_1048_gb300 as m
    return m


def _tuned(ovl, vol, key):
    f = getattr(ovl.lib, "_ZN3ovl18tuned_pair_variantEii")
    f.restype = ctypes.c_int
    return f(vol, key)


@pytest.mark.parametrize("dims,first", [((12, 12, 12, 12), "zero link"), ((12, 12, 12, 14), "su3")])
def test_shapes_are_tuned_by_route(ovl, dims, first):
    vol = int(np.prod(dims))
    ctx = ovl.ovl_ctx_create(0)
    lat = ovl.ovl_create_lattice(ctx, dims, -1)
    u = synth.gauge_links(dims, 61)
    cut = u.copy()
    cut.reshape(-1, 3, 3)[5] = 0  # no common scale: FP64 vectors
    b = torch.from_numpy(synth.gaussian_source(dims, 62)).cuda()
    x = torch.empty_like(b)
    p = ovl.ovl_sign_params_default(mu=0.3, fixed_k=4)
    ovl.ovl_set_pair_variant(vol, ovl.OVL_PREC_F64, -1)
    try:
        for name in (("zero link", "su3") if first == "zero link" else ("su3", "zero link")):
            ovl.ovl_set_links(lat, cut if name == "zero link" else u, ovl.OVL_F64)
            assert ovl.ovl_apply_sign(lat, p, b, x)[0] == ovl.OVL_OK
            keys = {k: _tuned(ovl, vol, k) for k in (FP64_VECTORS, FIXED_POINT)}
            if name == first:
                own, other = (FP64_VECTORS, FIXED_POINT) if name == "zero link" else (FIXED_POINT, FP64_VECTORS)
                assert keys[own] >= 0 and keys[other] == -1
                assert ovl.ovl_get_pair_variant(vol, ovl.OVL_PREC_F64) == keys[own]
        assert 0 <= keys[FP64_VECTORS] < 9 and keys[FIXED_POINT] in (0, 1)
        assert ovl.ovl_get_pair_variant(vol, ovl.OVL_PREC_F64) == keys[FIXED_POINT]
        ovl.ovl_set_pair_variant(vol, ovl.OVL_PREC_F64, 5)  # a pinned shape holds for both
        assert _tuned(ovl, vol, FP64_VECTORS) == _tuned(ovl, vol, FIXED_POINT) == 5
    finally:
        ovl.ovl_set_pair_variant(vol, ovl.OVL_PREC_F64, -1)
        ovl.ovl_destroy_lattice(lat)
        ovl.ovl_ctx_destroy(ctx)
    assert _tuned(ovl, vol, FP64_VECTORS) == _tuned(ovl, vol, FIXED_POINT) == -1
