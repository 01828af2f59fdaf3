"""D_W in FP64 on a field that does not fit fixed point (unit links), 12^4, eight sources: within twice the time that the
1368 flops a site take at the FP64 pipe's measured rate (180 us; 271 with every thread at work, 406 with three of four
idle)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

FP64_FLOPS = 1.256e12  # FMA chains on a GB300


def test_fields_beside_fixed_point_keep_the_fp64_rate():
    import paper_0910_1048_gb300 as ovl

    dims = (12, 12, 12, 12)
    ctx = ovl.ovl_ctx_create(0)
    lat = ovl.ovl_create_lattice(ctx, dims, -1)
    ovl.ovl_set_links(lat, synth.unit_links(dims), ovl.OVL_F64)
    inp = torch.from_numpy(synth.gaussian_source(dims, 81, nrhs=8)).cuda()
    out = torch.empty_like(inp)
    ts = []
    for _ in range(15):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        ovl.ovl_apply_DW(lat, -2.0, 0.3, 0, inp, out)
        b.record()
        torch.cuda.synchronize()
        ts.append(a.elapsed_time(b) * 1e-3)
    ovl.ovl_destroy_lattice(lat)
    ovl.ovl_ctx_destroy(ctx)
    assert np.median(ts[3:]) < 2 * 8 * 12 ** 4 * 1368 / FP64_FLOPS
