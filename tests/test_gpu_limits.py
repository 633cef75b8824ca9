"""Lattices at the limits of launches and memory, and calls after one that
failed: what is accepted there, and that nothing of a failed call stays."""
import gc

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


# The padded arrays of lattices whose rows are not 16-byte multiples (171 MB
# here) are there only while steps use them: no calls shorter than a chunk, no
# diagnostics at every step, not once the single pass is switched off; and they
# make room for what another allocation needs, also while the GPU still works on
# steps that use them.
def test_padded_arrays_only_where_steps_use_them(L, monkeypatch):
    import torch
    gc.collect()
    shape, size = (251, 64, 70), 2 * 19 * 252 * 64 * 70 * 4

    def held():
        torch.cuda.synchronize()
        return free - torch.cuda.mem_get_info()[0]

    def lattice(**options):
        lat = L.Lattice(*shape, 0.9, -5.5)
        for k, v in options.items():
            lat.set_option(k, v)
        lat.init_ligament(10.0, 251.0, 0.1, 0.3, 2.1, 0.1, 2.0)
        return lat

    with lattice(fused=0) as lat:
        lat.step(50)
        lat.sync()
        want = lat.rho()
    for options, calls, used in ((dict(diag_interval=1), (50,), False), (dict(diag_interval=20), (13, 26, 11), False),
                                 (dict(diag_interval=20), (13, 27, 10), True), (dict(), (1, 1, 48), True)):
        with lattice(**options) as lat:
            lat.diagnostics()
            torch.cuda.synchronize()
            free = torch.cuda.mem_get_info()[0]
            for n in calls:
                lat.step(n)
            assert (held() > size // 2) == used, (options, calls)
            lat.set_option("fused", 0)
            assert held() < size // 2
            np.testing.assert_array_equal(lat.rho(), want)

    with lattice() as lat:
        free = torch.cuda.mem_get_info()[0]
        lat.step(30)
        assert held() > size // 2
        monkeypatch.setenv("LBM_ALLOC_CAP_BYTES", str(size + (32 << 20)))
        lat.step(10)
        with L.Lattice(64, 64, 64, 0.9, -5.5, torch_buffers=False):     # 41 MB
            pass
        assert held() < size // 2
        lat.step(10)                                                    # on the two kernels
        np.testing.assert_array_equal(lat.rho(), want)
        monkeypatch.delenv("LBM_ALLOC_CAP_BYTES")
        lat.set_option("fused", 1)                                      # asked for again
        lat.step(2)
        assert held() > size // 2
