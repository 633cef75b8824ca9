"""Component labelling from both of its starts (the diagnostics pass over node
pairs and the labelling's own pass) at segment edges, and the diagnostics of
node pairs against one node per thread."""
import numpy as np
import pytest

import lbm_inputs
import oracle

pytestmark = pytest.mark.gpu

RL, RV = 2.65, 0.073


@pytest.fixture(scope="module")
def L():
    from paper_1904_11792_gb300 import build, lbm
    build.build()
    lbm.load()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return lbm


# even rows (pair start) shorter, equal and longer than its 64-node segments; odd rows and rows of less than a warp
SHAPES = [(62, 7, 5), (64, 6, 5), (66, 5, 6), (130, 4, 5), (200, 6, 4), (4, 9, 8), (37, 8, 7), (3, 5, 4), (65, 5, 5)]


@pytest.mark.parametrize("precision", ["f32", "f16dev", "f64"])
@pytest.mark.parametrize("p", [0.3, 0.6, 0.9])
@pytest.mark.parametrize("shape", SHAPES)
def test_labels_match_the_flood_fill(L, shape, p, precision):
    f = lbm_inputs.droplet_populations(*shape, seed=91, p=p, rho_l=RL, rho_v=RV)
    with L.Lattice(*shape, 1.0, -6.0, precision=precision, rho_ref=RV if precision == "f16dev" else 0.0) as lat:
        lat.set_option("rho_l", RL)
        lat.set_option("rho_v", RV)
        lat.set_populations(f)
        stored = lat.populations()
        d = lat.diagnostics(ccl=True)
        n, drops = lat.droplets()
    want_n, want = oracle.droplets(stored, RL, RV)
    sizes = [int(w[1]) for w in want]
    assert (d["droplets"], d["droplets_min8"], d["largest_droplet"]) == (want_n, sum(s >= 8 for s in sizes), max(sizes))
    assert n == want_n and [(g["first_node"], g["nodes"], g["x_slices"]) for g in drops] == [
        (int(w[0]), int(w[1]), int(w[10])) for w in want]


@pytest.mark.parametrize("mask", ["all", "rows", "planes", "snake"])
def test_labels_of_long_components(L, mask):
    nx, ny, nz = shape = (132, 12, 10)
    m = np.zeros((nz, ny, nx), bool)
    if mask == "all":
        m[:] = True
    elif mask == "rows":
        m[::2, ::2, :] = True
    elif mask == "planes":
        m[:, :, ::2] = True
    else:                       # one component winding through every other row of a plane, closed nowhere
        m[4, 0:11:2, :nx - 1] = True
        for k, y in enumerate(range(1, 10, 2)):
            m[4, y, (nx - 2) if k % 2 == 0 else 0] = True
    f = lbm_inputs.droplet_populations(*shape, seed=92, mask=m, rho_l=RL, rho_v=RV)
    with L.Lattice(*shape, 1.0, -6.0, precision="f32") as lat:
        lat.set_option("rho_l", RL)
        lat.set_option("rho_v", RV)
        lat.set_populations(f)
        stored = lat.populations()
        d = lat.diagnostics(ccl=True)
        n, drops = lat.droplets()
    want_n, want = oracle.droplets(stored, RL, RV)
    assert d["droplets"] == n == want_n
    assert [(g["first_node"], g["nodes"]) for g in drops] == [(int(w[0]), int(w[1])) for w in want]


@pytest.mark.parametrize("precision", ["f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("shape", [(62, 7, 5), (64, 16, 9), (130, 33, 20), (4, 9, 8)])
def test_pair_diagnostics_equal_single_node_diagnostics(L, shape, precision):
    """The same state from an array that starts at an odd element, which takes
    one node per thread: counts and extrema exact, sums to the rounding of two
    FP64 groupings of at most 2^14 terms."""
    import ctypes
    import torch
    nx, ny, nz = shape
    n, prec = nx * ny * nz, L.PRECISIONS[precision]
    dt = {"f32": torch.float32, "f16dev": torch.float16, "bf16dev": torch.bfloat16}[precision]
    f = lbm_inputs.random_populations(*shape, seed=93)
    out = []
    for first in (0, 1):
        buf = torch.zeros(19 * n + 1, dtype=dt, device="cuda")
        buf[first:first + 19 * n] = torch.from_numpy(f.reshape(-1)).to("cuda").to(dt)
        res = torch.zeros(13, dtype=torch.float64, device="cuda")
        rc = L.load().lbm_diagnostics_noalloc(ctypes.c_void_p(buf[first:].data_ptr()), nx, ny, nz, prec, 0.1, 2.0, 0.2,
                                              ctypes.c_void_p(res.data_ptr()), ctypes.c_void_p(0))
        assert rc == 0
        out.append(res.cpu().numpy())
    exact = [5, 7, 8, 9, 10, 11, 12]
    np.testing.assert_array_equal(out[0][exact], out[1][exact])
    np.testing.assert_allclose(out[0], out[1], rtol=1e-12, atol=1e-12 * out[0][0])
