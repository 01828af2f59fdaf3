"""The bench line's roofline of the FP64 direct method describes the kernel that runs: the fixed-point pair stencil, its
integer multiply-adds against the measured rate of that instruction, its bytes with the exponents."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def test_fixed_point_pair_stencil():
    infos = [[(0, [{"t_kernel_ms": 0.032, "kernel_samples": 4}])]]
    wl = bench.WORKLOADS["lattice12_mu0.3_direct_f64"]
    r = bench._roofline(wl, infos, 1.25, "probe", 9.0)
    t, vol = 0.032e-3, 12 ** 4
    # a hop: 9 link entries x 2 spins x 12 products; two stencils of eight; factors, diagonal, the dot
    mads = vol * (2 * 8 * 9 * 2 * 12 + 2 * 2 * 12 * 3 + 2 * 24 * 3 + 12 * 12)
    assert r["kernel"] == "k_fx_pair" and r["peak"] == 9.0 and r["bound"] == "alu"
    assert r["algorithmic_multiply_adds_per_launch"] == mads
    assert abs(r["achieved"] - mads / t / 1e12) < 1e-9 and abs(r["frac"] - r["achieved"] / 9.0) < 1e-12
    assert r["algorithmic_bytes_per_launch"] == vol * (576 + 4 * (192 + 4))
    # at mu = 0 the time hops have no factors
    assert bench.fx_pair_work(10, 3, False) == (10 * (576 + 3 * 4 * 196), 10 * 3 * (3456 + 144 + 144))
    # the other methods and precisions keep theirs
    assert bench._roofline(bench.WORKLOADS["lattice16_mu0.2_nrhs16_direct_f32"], infos, 1.25, "probe", 9.0)["bound"] == "hbm"
