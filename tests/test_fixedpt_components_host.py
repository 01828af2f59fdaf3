"""The FP64 stencil's fixed-point hop sums (csrc/fixedpt.cuh), built for the host, where components of a site or of
its neighbours differ in size: what FP64 arithmetic keeps of the small ones is kept."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import synth

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
