"""Small and thin lattices: the launch shapes chosen for rows shorter than a
warp, and the FP64 pseudo-potential's table at the edges of its ranges."""
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


@pytest.mark.parametrize("precision,pattern", [("f64", "ab"), ("f64", "aa"), ("f32", "aa"), ("f16dev", "ab")])
@pytest.mark.parametrize("shape", [(4, 49, 49), (3, 5, 70), (31, 9, 8), (62, 7, 3), (10, 3, 200), (66, 40, 9)])
def test_automatic_block_equals_explicit_block(L, shape, precision, pattern):
    f0 = lbm_inputs.random_populations(*shape, seed=71)
    out = []
    for block in (None, (32, 8, 1), (1, 1, 1)):
        with L.Lattice(*shape, 0.9, -5.5, precision=precision, pattern=pattern, block=block, rho_ref=0.1) as lat:
            lat.set_option("fused", 0)
            lat.set_populations(f0)
            lat.step(5)
            out.append(lat.populations())
    np.testing.assert_array_equal(out[0], out[1])
    np.testing.assert_array_equal(out[0], out[2])


def test_block_options_start_from_the_default_shape(L):
    with L.Lattice(4, 49, 49, 0.9, -5.5, precision="f32") as lat:
        assert [lat.get_option("block_" + k) for k in "xyz"] == [32, 8, 1]
        lat.set_option("block_x", 16)
        assert [lat.get_option("block_" + k) for k in "xyz"] == [16, 8, 1]


@pytest.mark.parametrize("rho0", [1.0, 1.7])
def test_f64_psi_against_expm1(L, rho0):
    """psi = rho0 (1 - exp(-rho / rho0)) within 2e-15 relative.  The table's
    Taylor series to the fourth power leaves d^5/720 of d, at most 1.3e-15 for
    d <= 1/256; three roundings and the entries' own (half a unit in the last
    place each) add at most 4.5e-16; from r = 8 on 1 - exp(-r) rounds once."""
    import torch
    k = np.arange(0, 2050) / 256.0
    edges = np.concatenate([k + s * e for e in (0.0, 1e-17, 1e-9, 1 / 512, 1 / 512 - 1e-12) for s in (-1, 1)])
    r = np.concatenate([edges, np.linspace(1e-6, 12.0, 5000), 2.0 ** -np.arange(1, 60), [8.0, np.nextafter(8.0, 0), 30.0]])
    r = np.unique(r[r > 0])
    shape = (12, 23, -(-r.size // (12 * 23)))     # x, y, z
    n = 12 * 23 * shape[2]
    rho = np.full(n, 1.0)
    rho[:r.size] = r * rho0
    f = np.zeros((19, n))
    f[0] = rho
    cfg = L.lbm_config_default()
    cfg.nx, cfg.ny, cfg.nz = shape
    cfg.G, cfg.rho0, cfg.precision = -5.5, rho0, L.LBM_F64
    sb, pb = L.lbm_required_bytes(cfg)
    psi = torch.empty(pb // 8, dtype=torch.float64, device="cuda")
    cfg.ext_psi, cfg.ext_psi_bytes = psi.data_ptr(), pb
    h = L.lbm_create_ex(cfg)
    try:
        L.lbm_set_populations(h, f)
        got_rho = L.lbm_moments(h, shape[::-1], ("rho",))["rho"].ravel()
        got = psi.cpu().numpy()
    finally:
        L.lbm_destroy(h)
    np.testing.assert_array_equal(got_rho, rho)
    want = -rho0 * np.expm1(-rho / rho0)
    assert np.max(np.abs(got - want) / want) <= 2e-15


@pytest.mark.parametrize("shape,precision,pattern,fused", [((64, 8, 12), "f32", "ab", 1), ((64, 8, 12), "f16dev", "ab", 1),
                                                           ((10, 9, 8), "f64", "ab", 0), ((12, 9, 8), "f16dev", "aa", 0)])
@pytest.mark.parametrize("interval", [0, 1, 3, 10])
def test_long_graphs_and_side_reductions_equal_eager_steps(L, shape, precision, pattern, fused, interval):
    """Small lattices replay longer graphs of chained launches, whose
    diagnostics are reduced beside the following steps: the state and every
    record equal those of single launches, over calls that mix both graph
    lengths and single steps."""
    f0 = lbm_inputs.random_populations(*shape, seed=72)
    out = []
    for graph in (1, 0):
        with L.Lattice(*shape, 0.9, -5.5, precision=precision, pattern=pattern, rho_ref=0.1) as lat:
            lat.set_option("fused", fused)
            lat.set_option("graph", graph)
            lat.set_option("rho_l", 2.0)
            lat.set_option("rho_v", 0.2)
            lat.set_option("diag_interval", interval)
            lat.set_populations(f0)
            recs = []
            for n in (40, 7, 23, 60):
                lat.step(n)
                recs += lat.diag_history()
            lat.sync()
            out.append((lat.populations(), recs))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1]
    assert [r["step"] for r in out[0][1]] == ([] if not interval else list(range(0, 130, interval)))


@pytest.mark.parametrize("shape", [(37, 11, 9), (96, 96, 64), (160, 128, 110)])   # 19, 14 and 3 planes cross at a time
def test_host_transfers_in_groups_of_planes(L, shape):
    nx, ny, nz = shape
    rng = np.random.default_rng(73)
    f0 = rng.uniform(0.01, 0.1, (19, nz, ny, nx))
    with L.Lattice(*shape, 0.9, -5.5, precision="f64") as lat:
        lat.set_populations(f0)
        np.testing.assert_array_equal(lat.populations(), f0)
        every = lat.moments()      # all four fields together, except on the largest shape
        for k, v in every.items():
            np.testing.assert_array_equal(lat.moments((k,))[k], v)
    np.testing.assert_allclose(every["rho"], f0.sum(axis=0), rtol=1e-14)


def test_diag_history_across_the_ring_end(L):
    """More records than the ring's 1024 slots, read in two calls: the second
    one's slots wrap around the ring's end."""
    f0 = lbm_inputs.random_populations(8, 5, 4, seed=74)
    with L.Lattice(8, 5, 4, 0.9, -5.5, precision="f64") as lat:
        lat.set_option("diag_interval", 1)
        lat.set_populations(f0)
        lat.step(1000)
        a = lat.diag_history()
        lat.step(100)
        b = lat.diag_history()
        lat.step(30)
        c = lat.diag_history(7)
        d = lat.diagnostics()
    assert [r["step"] for r in a + b] == list(range(1100)) and [r["step"] for r in c] == list(range(1123, 1130))
    assert all(abs(r["mass"] / d["mass"] - 1) < 1e-11 for r in a + b + c)


@pytest.mark.parametrize("precision", ["f32", "f16dev"])
def test_small_lattices_take_the_two_kernels_until_asked(L, precision):
    shape, f0 = (64, 8, 12), lbm_inputs.random_populations(64, 8, 12, seed=75)
    out = []
    for option in (None, ("fused", 1), ("fused_fz", 4), ("fused_group", 1)):
        with L.Lattice(*shape, 0.9, -5.5, precision=precision, rho_ref=0.1) as lat:
            assert lat.get_option("fused") == 1
            if option:
                lat.set_option(*option)
            lat.set_option("kernel_timing", 1)
            lat.set_populations(f0)
            lat.step(3)
            assert [L.lbm_kernel_time(lat.h, k)[0] for k in range(3)] == ([0, 0, 3] if option else [3, 3, 0])
            out.append(lat.populations())
    for f in out[1:]:
        np.testing.assert_array_equal(out[0], f)


@pytest.mark.parametrize("precision", ["f16dev", "bf16dev"])
@pytest.mark.parametrize("rounding", [0, 1])
@pytest.mark.parametrize("shape,blocks", [((64, 64, 64), 2), ((128, 128, 128), 2), ((130, 128, 127), 3)])
def test_two_byte_pairs_round_as_single_nodes(L, shape, blocks, rounding, precision):
    """The rounding bits of two nodes taken at once, and the two-kernel step's
    blocks per SM either side of 2^21 nodes: bitwise the one-node kernels."""
    f0 = lbm_inputs.random_populations(*shape, seed=72)
    out = []
    for vector, fused in ((1, 0), (0, 0), (1, 1)):
        with L.Lattice(*shape, 0.9, -5.5, precision=precision, rho_ref=0.1) as lat:
            lat.set_option("fused", fused if shape[0] % 64 == 0 else 0)
            lat.set_option("vector", vector)
            lat.set_option("stochastic_rounding", rounding)
            if vector and not fused:
                assert lat.get_option("occupancy") == blocks
            lat.set_populations(f0)
            lat.step(5)
            out.append(lat.populations())
    np.testing.assert_array_equal(out[0], out[1])
    np.testing.assert_array_equal(out[0], out[2])
