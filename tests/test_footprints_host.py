"""Device memory a request is charged for, against the arrays a solve allocates (sizes in bytes per source)."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def lib():
    import paper_0910_1048_gb300 as ovl

    direct = getattr(ovl.lib, "_ZN3ovl16direct_footprintEiiibb")
    multi = getattr(ovl.lib, "_ZN3ovl20multishift_footprintEiiibb")
    for f, flags in ((direct, 2), (multi, 2)):
        f.restype = ctypes.c_size_t
        f.argtypes = [ctypes.c_int] * 3 + [ctypes.c_bool] * flags
    return direct, multi


SLOTS = 256  # partial-sum slots above one per 128 elements
DEFL = 16    # deflation vectors whose partial sums are provided for


def _slots(vol):
    return (12 * vol + 127) // 128 + SLOTS


@pytest.mark.parametrize("vol,nrhs", [(256, 1), (20736, 1), (20736, 64), (65536, 16), (1 << 20, 4)])
@pytest.mark.parametrize("f64", [True, False])
@pytest.mark.parametrize("two_pass", [True, False])
def test_direct(lib, vol, nrhs, f64, two_pass):
    kmax, elt, vec = 300, 16 if f64 else 8, 12 * vol
    columns = 3 if two_pass else kmax + 1
    need = columns * vec * elt + 4 * vec * elt  # basis; what_j, what_{j-1}, A v, A w
    need += 3 * vec * 16 + (vec * 16 if two_pass else 0)  # x_P, staged b and x, the second pass's sum
    need += DEFL * _slots(vol) * 32  # partial sums
    if f64:
        need += 6 * 4 * vol + 256  # exponents of the six fixed-point vectors, the step's coefficients
    got = lib[0](vol, nrhs, kmax, f64, two_pass)
    assert nrhs * need <= got <= 1.001 * nrhs * need + (2 << 20)


@pytest.mark.parametrize("vol,nrhs,s", [(256, 1, 4), (20736, 1, 20), (65536, 4, 20), (65536, 16, 80)])
@pytest.mark.parametrize("f64,refine", [(True, False), (False, False), (False, True)])
def test_multishift(lib, vol, nrhs, s, f64, refine):
    elt, vec = 16 if f64 else 8, 12 * vol
    need = nrhs * (6 * vec * elt + s * vec * elt + 5 * vec * 16 + DEFL * _slots(vol) * 32)
    if refine:  # x^(i), r, and up to 1024 corrections: four FP64 vectors, six FP32 ones, their sum, partial sums
        systems = min(1024, nrhs * s)
        need += nrhs * (s + 1) * vec * 16 + systems * (vec * (4 * 16 + 6 * 8 + 16) + _slots(vol) * 32)
    got = lib[1](vol, nrhs, s, f64, refine)
    assert need <= got <= 1.001 * need + (2 << 20)
