"""The FP64 stencil's fixed-point hop sums (csrc/fixedpt.cuh), built for the host, against the same sums in
extended precision.

Bound per component, with S the power of two of the common scale (at most four times the largest neighbour
component times max(1, e^|mu|)): per hop the cut of the spinor limbs (2 x 2.45 / 2 units of 2^-58 S), the rounded
links (3), the dropped low products (12) and the rounding of the cross sum (1), at most 20.5 units with the
shifts, over eight hops 164 < 2^8 units and factors below 4 on two of them: 2^-49 S |hop coefficient| times
the links' scale; then three FP64 roundings (the unit, the conversion and the final fused multiply-add).
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import synth

HERE = os.path.dirname(os.path.abspath(__file__))
DIMS = (4, 6, 2, 8)
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


def _check(lib, u, psi, mu=0.3, g5=0, t_bc=-1):
    v = int(np.prod(DIMS))
    d = np.array(DIMS, np.int32)
    un = np.ascontiguousarray(u.reshape(4, v, 9).transpose(0, 2, 1))
    pn = np.ascontiguousarray(psi.reshape(v, 12).T)
    fx, f64, efx, ef64 = [np.zeros((12, v, 2)) for _ in range(4)]
    usable = np.zeros(v, np.int32)
    ok = lib.dslash_check(d.ctypes.data, t_bc, -2.0, mu, g5, un.ctypes.data, pn.ctypes.data, fx.ctypes.data,
                          f64.ctypes.data, efx.ctypes.data, ef64.ctypes.data, usable.ctypes.data)
    return bool(ok), fx, efx, ef64, usable


def _nb_max(psi):
    """Largest component among a site's eight neighbours: [V]."""
    lx, ly, lz, lt = DIMS
    a = np.maximum(np.abs(psi.real), np.abs(psi.imag)).reshape(lt, lz, ly, lx, 12).max(-1)
    m = np.zeros_like(a)
    for ax in range(4):
        for sh in (1, -1):
            m = np.maximum(m, np.roll(a, sh, ax))
    return m.ravel()


def _bound(psi, fx, mu, scale=1.0):
    v = int(np.prod(DIMS))
    own = np.abs(psi.reshape(v, 12).T.copy().view(np.float64).reshape(12, v, 2))
    hop = 2.0 ** -49 * 4 * _nb_max(psi) * max(1.0, np.exp(abs(mu))) * KAPPA * scale
    return hop[None, :, None] + 2.0 ** -53 * (3 * np.abs(fx) + 2 * own)


@pytest.mark.parametrize("mu", [0.0, 0.3, -0.3, 1.4, -5.0, 16.0])
@pytest.mark.parametrize("g5,t_bc", [(0, -1), (1, 1)])
def test_hop_sums(lib, mu, g5, t_bc):
    u, psi = synth.gauge_links(DIMS, 1), synth.gaussian_source(DIMS, 2)
    ok, fx, efx, ef64, usable = _check(lib, u, psi, mu, g5, t_bc)
    assert ok and usable.all()
    assert (efx <= _bound(psi, fx, mu)).all()
    # the typical error: the FP64 roundings at the end, at most 2^-52 of the output together
    assert np.linalg.norm(efx) <= 2.0 ** -52 * np.linalg.norm(fx)


@pytest.mark.parametrize("spread", [3.0, 40.0, 300.0])
def test_sites_of_different_size(lib, spread):
    """The scale is the neighbourhood's own: fields whose sites differ by up to e^300."""
    u, psi = synth.gauge_links(DIMS, 1), synth.gaussian_source(DIMS, 2)
    lx, ly, lz, lt = DIMS
    w = np.exp(np.random.default_rng(3).uniform(-spread, spread, (lt, lz, ly, lx, 1, 1)))
    ok, fx, efx, _, usable = _check(lib, u, psi * w)
    assert ok and usable.all()
    assert (efx <= _bound(psi * w, fx, 0.3)).all()


@pytest.mark.parametrize("scale", [0.01, 1.0 + 1e-12, 3.0, 200.0])
def test_scaled_links(lib, scale):
    u, psi = synth.gauge_links(DIMS, 4) * scale, synth.gaussian_source(DIMS, 5)
    ok, fx, efx, _, usable = _check(lib, u, psi)
    assert ok and usable.all()
    assert (efx <= _bound(psi, fx, 0.3, 4 * scale)).all()  # (the field's scale is a power of two above it)


def _broken(kind):
    u = synth.gauge_links(DIMS, 4).copy()
    one = u.reshape(-1, 3, 3)[37]
    if kind == "zero link":
        one[:] = 0
    if kind == "small link":
        one *= 1e-3
    if kind == "nan":
        one[1, 2] = np.nan
    if kind == "inf":
        one[0, 0] = np.inf
    if kind == "huge":
        u *= 1e5
    if kind == "tiny":
        u *= 1e-5
    return u


@pytest.mark.parametrize("kind", ["zero link", "small link", "nan", "inf", "huge", "tiny"])
def test_fields_without_a_common_scale_are_refused(lib, kind):
    assert not _check(lib, _broken(kind), synth.gaussian_source(DIMS, 5))[0]


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_sites_beside_a_non_finite_value_are_refused(lib, value):
    u, psi = synth.gauge_links(DIMS, 1), synth.gaussian_source(DIMS, 2)
    lx, ly, lz, lt = DIMS
    mark = np.zeros((lt, lz, ly, lx), bool)
    mark[5, 1, 2, 3] = True
    psi[5, 1, 2, 3, 2, 1] = value
    want = np.zeros_like(mark)
    for ax in range(4):
        for sh in (1, -1):
            want |= np.roll(mark, sh, ax)
    usable = _check(lib, u, psi)[4].astype(bool)
    assert (usable == ~want.ravel()).all()


def test_small_values(lib):
    """All zero is exact; components all below 2^-959 are refused."""
    u, psi = synth.gauge_links(DIMS, 1), synth.gaussian_source(DIMS, 2)
    ok, fx, efx, _, usable = _check(lib, u, 0 * psi)
    assert usable.all() and not fx.any()
    assert not _check(lib, u, 1e-300 * psi)[4].any()
    assert not _check(lib, u, psi, mu=16.5)[4].any()
