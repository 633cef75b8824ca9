"""The single pass on small lattices, which take the two kernels until it is
asked for: checks of test_gpu_parity.py and test_gpu_droplets.py that step such
lattices with the options' defaults, with it."""
import pytest

import test_gpu_droplets as droplets
import test_gpu_parity as parity

pytestmark = pytest.mark.gpu

L, coex = parity.L, parity.coex


@pytest.fixture(autouse=True)
def single_pass(L, monkeypatch):
    """Every lattice that the single pass applies to is asked for it, and has to
    have run it when it is closed."""
    create, close = L.Lattice.__init__, L.Lattice.close
    seen = []

    def asked(lat, *args, **kw):
        create(lat, *args, **kw)
        lat.asked = lat.get_option("fused") == 1
        if lat.asked:
            lat.set_option("fused", 1)
            seen.append(lat.shape)

    def checked(lat):
        if getattr(lat, "h", None) and lat.asked and lat.step_count:
            lat.set_option("kernel_timing", 1)
            lat.step(3)
            assert [L.lbm_kernel_time(lat.h, k)[0] for k in range(3)] == [0, 0, 3]
        close(lat)

    monkeypatch.setattr(L.Lattice, "__init__", asked)
    monkeypatch.setattr(L.Lattice, "close", checked)
    yield
    assert seen


@pytest.mark.parametrize("precision", ["f32", "f16dev"])
@pytest.mark.parametrize("shape,k", [((64, 16, 12), 4), ((128, 8, 17), 3), ((64, 8, 3), 1)])
def test_diagnostics_in_the_pass(L, coex, precision, shape, k):
    parity.test_fused_diag_history_matches_on_demand(L, coex, precision, shape, k)


@pytest.mark.parametrize("precision", ["f32", "f16dev"])
def test_checkpoint(L, coex, precision):
    parity.test_checkpoint_resume_bitwise(L, coex, "ab", precision, 64)


@pytest.mark.parametrize("precision", ["f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("k", [0, 3])
def test_graphs(L, precision, k):
    parity.test_graph_equals_eager_bitwise(L, "ab", precision, (64, 8, 10), k)


def test_oracle_ligament(L, coex):
    parity.test_fp32_ligament_parity_100_steps(L, coex, "ab")


@pytest.mark.parametrize("precision,tol", [("f16dev", 5e-3), ("bf16dev", 4e-2)])
def test_deviation_storage(L, coex, precision, tol):
    parity.test_deviation_storage_error(L, coex, precision, tol)


def test_fp32_drift(L, coex):
    parity.test_fp64_mass_resolves_fp32_drift(L, coex)


@pytest.mark.parametrize("precision,tol", [("f16dev", 1e-5), ("bf16dev", 3e-4)])
def test_rounding_drift(L, coex, precision, tol):
    parity.test_stochastic_rounding_mass_drift(L, coex, precision)
    parity.test_uniform_liquid_keeps_its_mass(L, coex, precision, tol)


def test_droplet_counts(L):
    droplets.test_droplet_counts_inside_the_time_loop(L)
