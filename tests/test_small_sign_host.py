"""sign(H_k) e_1 on the host: what its result must not depend on."""
import numpy as np
import pytest

import synth
from oracle import deflation, lanczos

DIMS = (4, 4, 4, 4)


@pytest.fixture(scope="module")
def ovl():
    import paper_0910_1048_gb300 as m
    return m


@pytest.fixture(scope="module")
def h800():
    """H_k of two-sided Lanczos at 4^4, mu = 0.3, k = 800 (its leading blocks are the smaller ones)."""
    u, b = synth.gauge_links(DIMS, 3), synth.gaussian_source(DIMS, 4)
    a, ah = deflation.sparse_hw(u, DIMS, -2.0, 0.3), deflation.sparse_hw(u, DIMS, -2.0, -0.3)
    _, st = lanczos.direct_lanczos_lr(lambda v: (a @ v.ravel()).reshape(v.shape),
                                      lambda w: (ah @ w.ravel()).reshape(w.shape), b, 800)
    return st["alpha"], st["beta"], st["delta"]


def _block(h, k):
    return h[0][:k], h[1][:k - 1], h[2][:k - 1]


@pytest.mark.parametrize("k", [40, 200, 400, 800])
def test_result_does_not_depend_on_the_threads(ovl, h800, k):
    """The shifts are summed in parts that (s, k) alone decide: evaluations that share the host's threads (a batch's
    sources) give the same bits as one that has them all."""
    share = getattr(ovl.lib, "_ZN3ovl20set_sign_concurrencyEi")
    try:
        ys = []
        for n in (1, 2, 3, 64):
            share(n)
            st, y = ovl.ovl_small_sign(*_block(h800, k))
            assert st == ovl.OVL_OK
            ys.append(y)
    finally:
        share(1)
    assert all(np.array_equal(y, ys[0]) for y in ys)


@pytest.mark.parametrize("method", [0, 1, 2, 3])
@pytest.mark.parametrize("k", [12, 60, 200, 400])
def test_large_and_tiny_matrices(ovl, h800, k, method):
    """sign(c H) = sign(H) for c > 0: the same status and result, by a power of two to the last bits, and never
    OK with numbers that are not finite. 1e-9: the routes' own checks."""
    if method == 2 and k > 60:
        pytest.skip("dense Newton: O(k^3) a step")
    h = _block(h800, k)
    st, y = ovl.ovl_small_sign(*h, method)
    for c in (2.0 ** -900, 2.0 ** -480, 1e-200, 1e-140, 1e140, 1e200, 2.0 ** 480, 2.0 ** 900):
        stc, yc = ovl.ovl_small_sign(*(c * a for a in h), method)
        assert stc == st, c
        if st == ovl.OVL_OK:
            assert np.linalg.norm(yc - y) <= 1e-9 * np.linalg.norm(y), c
            if np.log2(c) == round(np.log2(c)) and method != 2:
                assert np.linalg.norm(yc - y) <= 1e-12 * np.linalg.norm(y), c


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_matrices_that_are_not_finite(ovl, h800, bad):
    for n in (5, 60):
        for part in range(3):
            h = [a.copy() for a in _block(h800, n)]
            h[part][n // 2] = bad
            st, y = ovl.ovl_small_sign(*h)
            assert st != ovl.OVL_OK or np.isfinite(y).all()
