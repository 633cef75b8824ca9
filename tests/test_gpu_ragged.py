"""The single-pass step on lattices that the 64-wide tiles do not divide: on the
lattice's own rows where they are 16-byte multiples, on padded copies inside
replayed chunks of steps otherwise.  Both equal the two-kernel step bitwise."""
import numpy as np
import pytest

import lbm_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1904_11792_gb300 import build, lbm
    build.build()
    lbm.load()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return lbm


# rows of 4 k (direct for FP32), 8 k (direct for 2-byte storage too), even and odd lengths; one and several tiles
# per row, rows ending one node into a tile, heights around the tile rows
SHAPES = [(251, 12, 11), (100, 13, 9), (66, 16, 9), (32, 17, 10), (129, 5, 12), (200, 9, 8), (192, 10, 7), (5, 3, 4), (8, 3, 3)]


@pytest.mark.parametrize("precision,mrt", [("f32", 0), ("f16dev", 0), ("bf16dev", 0), ("f32", 1), ("f16dev", 1)])
@pytest.mark.parametrize("shape", SHAPES)
def test_ragged_step_equals_two_kernel_step(L, shape, precision, mrt):
    f0 = lbm_inputs.random_populations(*shape, seed=81)
    out = []
    for fused in (2, 0):     # 2: whatever the lattice's size
        with L.Lattice(*shape, 0.9, -5.5, precision=precision, rho_ref=0.1) as lat:
            lat.set_option("fused", fused)
            lat.set_option("collision", mrt)
            lat.set_populations(f0)
            got = []
            for n in (1, 2, 5, 23):
                lat.step(n)
                got.append(lat.populations())
            lat.sync()
            out.append(got)
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("precision", ["f32", "f16dev"])
@pytest.mark.parametrize("interval,ccl", [(1, 0), (2, 0), (10, 0), (10, 1)])
@pytest.mark.parametrize("shape", [(251, 12, 11), (100, 13, 9)])
def test_ragged_step_with_diagnostics(L, shape, precision, interval, ccl):
    f0 = lbm_inputs.random_populations(*shape, seed=82)
    out = []
    for fused, graph in ((2, 1), (2, 0), (0, 1)):
        with L.Lattice(*shape, 0.9, -5.5, precision=precision, rho_ref=0.1) as lat:
            for k, v in (("fused", fused), ("graph", graph), ("rho_l", 2.0), ("rho_v", 0.2), ("diag_ccl", ccl),
                         ("diag_interval", interval)):
                lat.set_option(k, v)
            lat.set_populations(f0)
            recs = []
            for n in (20, 3, 27):
                lat.step(n)
                recs += lat.diag_history()
            out.append((lat.populations(), recs))
    for f, recs in out[1:]:
        np.testing.assert_array_equal(out[0][0], f)
        assert out[0][1] == recs


def test_ragged_step_is_the_default_on_larger_lattices(L):
    """Above 2^20 nodes kernel timing counts single passes; the option's value
    keeps naming the 64-wide tiles only."""
    for shape, want in (((172, 80, 80), 4), ((100, 13, 9), 0)):
        with L.Lattice(*shape, 1.0, -6.0, precision="f32") as lat:
            assert lat.get_option("fused") == 0
            lat.init_ligament(12.0, float(shape[0]), 0.02, 0.0, 2.6489, 0.0732, 2.0)
            lat.set_option("kernel_timing", 1)
            lat.step(4)
            assert L.lbm_kernel_time(lat.h, 2)[0] == want


@pytest.mark.parametrize("shape,srt,mrt", [((576, 80, 83), 9, 17), ((128, 96, 101), 12, 11), ((64, 8, 5), 4, 4)])
def test_run_length_follows_the_collision(L, shape, srt, mrt):
    """The single pass chooses its run length by the collision; its bits, the
    diagnostics' scratch and the switch between them do not depend on it."""
    out = []
    for fused in (1, 0):
        with L.Lattice(*shape, 0.95, -5.3, precision="f32") as lat:
            lat.init_ligament(min(shape[1:]) / 4.0, float(shape[0]), 0.1, 0.3, 2.1085, 0.0778, 2.0)
            lat.set_option("fused", fused)
            lat.set_option("diag_interval", 3)
            for collision, fz in ((1, mrt), (0, srt), (1, mrt)):
                lat.set_option("collision", collision)
                assert lat.get_option("fused_fz_used") == fz
                lat.step(4)
            lat.sync()
            out.append((lat.populations(), [d["mass"] for d in lat.diag_history()]))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_allclose(out[0][1], out[1][1], rtol=1e-13)   # FP64 sums of N < 2^22 terms
