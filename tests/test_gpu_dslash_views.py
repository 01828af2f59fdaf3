"""Native FP32 batches in views that start on 8 bytes, on a field whose links (74 MB) do not stay in L2: the sources share
them as in an aligned batch, with the same bits."""
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nrhs", [2, 5])
def test_native_batch_in_a_view_of_8_bytes(nrhs):
    import paper_0910_1048_gb300 as ovl

    dims = (22, 22, 22, 24)
    ctx = ovl.ovl_ctx_create(0)
    lat = ovl.ovl_create_lattice(ctx, dims, -1)
    tile = synth.gauge_links((22, 22, 2, 2), 71)  # repeated along z and t: any links will do
    ovl.ovl_set_links(lat, tile.repeat(12, 1).repeat(11, 2), ovl.OVL_F32)
    n = nrhs * 12 * 22 * 22 * 22 * 24
    gen = torch.Generator(device="cuda")
    gen.manual_seed(72)
    psi = torch.view_as_complex(torch.randn((n, 2), dtype=torch.float32, device="cuda", generator=gen)).view(
        nrhs, 24, 22, 22, 22, 4, 3)
    for dagger in (0, ovl.OVL_DAGGER):
        flags = ovl.OVL_NATIVE | ovl.OVL_GAMMA5 | ovl.OVL_LINKS_F32 | dagger
        want = torch.empty_like(psi)
        ovl.ovl_apply_DW(lat, -2.0, 0.3, flags, psi, want)
        for oi, oo in ((1, 0), (0, 1), (1, 1)):
            a, b = (torch.full((n + 2,), float("nan"), dtype=torch.complex64, device="cuda") for _ in range(2))
            src, got = a[oi:oi + n].view(psi.shape), b[oo:oo + n].view(psi.shape)
            assert (src.data_ptr() % 16, got.data_ptr() % 16) == (8 * oi, 8 * oo)
            src.copy_(psi)
            ovl.ovl_apply_DW(lat, -2.0, 0.3, flags, src, got)
            assert torch.equal(torch.view_as_real(got), torch.view_as_real(want))
            assert torch.isnan(torch.cat([b[:oo], b[oo + n:]]).real).all()  # nothing beside the view is written
    ovl.ovl_destroy_lattice(lat)
    ovl.ovl_ctx_destroy(ctx)
