"""The fixed-point copy of the links: made by ovl_set_links for callers that name FP64, at the first FP64 use for the
others, never in a capture."""
import threading

import numpy as np
import pytest

import synth
from oracle import krylov, wilson

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DIMS = (6, 4, 4, 8)


@pytest.fixture(scope="module")
def ovl():
    import paper_0910_1048_gb300 as m
    return m


@pytest.fixture(scope="module")
def ctx(ovl):
    c = ovl.ovl_ctx_create(0)
    yield c
    ovl.ovl_ctx_destroy(c)


def _close(got, u, psi):
    ref = wilson.apply_dw(u, psi, -2.0, 0.3, -1)
    assert np.abs(got.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()


def test_reduced_formats_hold_no_copy(ovl, ctx):
    """24^4, 191 MB a copy: FP64 and FP32 links without it, with it after an FP64 operator."""
    dims = (24, 24, 24, 24)
    tile = synth.gauge_links((24, 24, 2, 2), 1)
    u = torch.from_numpy(np.ascontiguousarray(tile.repeat(12, 1).repeat(12, 2))).cuda()
    psi = torch.randn(12 * 24 ** 4, dtype=torch.complex128, device="cuda")
    out = torch.empty_like(psi)
    torch.cuda.synchronize()
    held = []
    lat = ovl.ovl_create_lattice(ctx, dims, -1)
    free = torch.cuda.mem_get_info()[0]
    for step in (lambda: ovl.ovl_set_links(lat, u, ovl.OVL_F32), lambda: ovl.ovl_apply_DW(lat, -2.0, 0.3, 0, psi, out),
                 lambda: ovl.ovl_apply_DW(lat, -2.0, 0.3, 0, psi, out)):
        step()
        torch.cuda.synchronize()
        held.append((free - torch.cuda.mem_get_info()[0]) / (24 ** 4 * 288))
    ovl.ovl_destroy_lattice(lat)
    assert abs(held[0] - 3) < 0.2 and abs(held[1] - 5) < 0.2 and held[2] == held[1]


def test_first_use_by_two_threads(ovl, ctx):
    u, psi = synth.gauge_links(DIMS, 2), synth.gaussian_source(DIMS, 3, nrhs=2)
    for _ in range(4):
        lat = ovl.ovl_create_lattice(ctx, DIMS, -1)
        ovl.ovl_set_links(lat, u, ovl.OVL_F32)
        inp = torch.from_numpy(psi).cuda()
        outs = [torch.empty_like(inp[0]) for _ in range(2)]
        torch.cuda.synchronize()
        go = threading.Barrier(2)

        def work(r):
            with torch.cuda.stream(torch.cuda.Stream()):
                go.wait()
                ovl.ovl_apply_DW(lat, -2.0, 0.3, 0, inp[r], outs[r])
                torch.cuda.current_stream().synchronize()

        th = [threading.Thread(target=work, args=(r,)) for r in range(2)]
        for t in th:
            t.start()
        for t in th:
            t.join()
        for r in range(2):
            _close(outs[r], u, psi[r])
        ovl.ovl_destroy_lattice(lat)


def test_capture_before_the_copy(ovl, ctx):
    """An FP64 operator captured on a lattice without the copy stays right when the copy and other links come."""
    u, u2, psi = synth.gauge_links(DIMS, 4), synth.gauge_links(DIMS, 5), synth.gaussian_source(DIMS, 6)
    lat = ovl.ovl_create_lattice(ctx, DIMS, -1)
    ovl.ovl_set_links(lat, u, ovl.OVL_F32)
    inp = torch.from_numpy(psi).cuda()
    out = torch.empty_like(inp)
    graph, st = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=st):
        ovl.ovl_apply_DW(lat, -2.0, 0.3, 0, inp, out)
    graph.replay()
    torch.cuda.synchronize()
    _close(out, u, psi)
    direct = torch.empty_like(inp)
    ovl.ovl_apply_DW(lat, -2.0, 0.3, 0, inp, direct)  # makes the copy
    torch.cuda.synchronize()
    _close(direct, u, psi)
    for links in (u2, synth.unit_links(DIMS), u):
        ovl.ovl_set_links(lat, links, ovl.OVL_F64)
        out.zero_()
        graph.replay()
        ovl.ovl_apply_DW(lat, -2.0, 0.3, 0, inp, direct)
        torch.cuda.synchronize()
        _close(out, links, psi)
        _close(direct, links, psi)
    ovl.ovl_destroy_lattice(lat)


@pytest.mark.parametrize("formats", ["f32", "f32 then f64", "f64"])
def test_solves_whatever_the_formats(ovl, ctx, formats):
    """FP64 direct at equal k: the same bits once the copy is there, and Algorithm 4 to 1e-10."""
    u, b, k = synth.gauge_links(DIMS, 7), synth.gaussian_source(DIMS, 8), 20
    lat = ovl.ovl_create_lattice(ctx, DIMS, -1)
    if formats != "f64":
        ovl.ovl_set_links(lat, u, ovl.OVL_F32)
    if formats != "f32":
        ovl.ovl_set_links(lat, u, ovl.OVL_F64)
    bt = torch.from_numpy(b).cuda()
    p = ovl.ovl_sign_params_default(mu=0.3, fixed_k=k, check_every=6)
    xs = [torch.empty_like(bt) for _ in range(3)]
    assert ovl.ovl_apply_sign(lat, p, bt, xs[0])[0] == ovl.OVL_OK
    assert ovl.ovl_apply_sign_noalloc(lat, p, bt, xs[1])[0] == ovl.OVL_OK
    assert ovl.ovl_apply_sign(lat, p, bt, xs[2])[0] == ovl.OVL_OK
    ovl.ovl_destroy_lattice(lat)
    xo, _, _ = krylov.direct_lanczos(u, DIMS, -2.0, 0.3, b, k)
    for x in xs:
        x = x.cpu().numpy()
        assert np.linalg.norm(x - xo) < 1e-10 * np.linalg.norm(xo)
    assert torch.equal(torch.view_as_real(xs[0]), torch.view_as_real(xs[2]))


def test_allocation_free_solve_without_the_copy(ovl, ctx):
    u, b, k = synth.gauge_links(DIMS, 9), synth.gaussian_source(DIMS, 10), 20
    lat = ovl.ovl_create_lattice(ctx, DIMS, -1)
    ovl.ovl_set_links(lat, u, ovl.OVL_F32)
    bt = torch.from_numpy(b).cuda()
    x = torch.empty_like(bt)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    assert ovl.ovl_apply_sign_noalloc(lat, ovl.ovl_sign_params_default(mu=0.3, fixed_k=k), bt, x)[0] == ovl.OVL_OK
    assert torch.cuda.mem_get_info()[0] >= free - (4 << 20)
    ovl.ovl_destroy_lattice(lat)
    xo, _, _ = krylov.direct_lanczos(u, DIMS, -2.0, 0.3, b, k)
    assert np.linalg.norm(x.cpu().numpy() - xo) < 1e-10 * np.linalg.norm(xo)
