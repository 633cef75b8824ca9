"""The autotuner's choices for a lattice are no slower than what the library runs untuned."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1904_11792_gb300 import build, lbm
    build.build()
    lbm.load()
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return lbm


def step_us(obj, steps, reps=5):
    import torch
    best = float("inf")
    for _ in range(reps + 1):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        obj.step(steps)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, 1e3 * e0.elapsed_time(e1) / steps)
    return best


# Rows the tiles do not divide (the single pass runs in replayed graphs), rows
# shorter than a warp (blocks of several rows), and in place (a register budget
# of its own for odd steps): the choice is the library's own, or as fast within
# a tenth of it.
@pytest.mark.parametrize("shape,precision,pattern", [((251, 112, 112), "f32", "ab"), ((4, 49, 49), "f64", "ab"),
                                                     ((256, 96, 96), "f16dev", "aa")])
def test_tuned_lattice_is_no_slower_than_untuned(L, shape, precision, pattern):
    from paper_1904_11792_gb300 import autotune
    choice = autotune.tune_lattice(*shape, precision=precision, patterns=(pattern,), use_cache=False)
    assert choice["pattern"] == pattern
    us = []
    for tuned in (False, True):
        with L.Lattice(*shape, 1.0, -6.0, precision=precision, pattern=pattern,
                       rho_ref=0.0732 if precision == "f16dev" else 0.0) as lat:
            if tuned:
                autotune.apply(lat, choice)
            lat.init_ligament(shape[1] / 4.0, float(shape[0]), 0.02, 0.0, 2.6489, 0.0732, 2.0)
            us.append(step_us(lat, 64))
            lat.sync()
    assert us[1] <= 1.1 * us[0], (us, choice)
