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


# Caller's buffers that start at any element: refused by the single pass (its
# copies want 16 bytes; on small lattices too, which take the two kernels by
# default), stepped by the two kernels one node at a time where pairs or groups
# of four nodes would be misaligned.  Off its elements a buffer is refused.
@pytest.mark.parametrize("precision,pattern", [("f64", "ab"), ("f32", "ab"), ("f32", "aa"), ("f16dev", "ab"),
                                               ("f16dev", "aa"), ("bf16dev", "ab")])
@pytest.mark.parametrize("shape", [(64, 8, 12), (66, 7, 9), (61, 7, 9)])
def test_buffers_at_any_element(L, shape, precision, pattern):
    import torch
    f0 = lbm_inputs.random_populations(*shape, seed=97)
    cfg = L.lbm_config_default()
    cfg.nx, cfg.ny, cfg.nz = shape
    cfg.tau, cfg.G, cfg.rho_ref = 0.9, -5.5, 0.1
    cfg.precision, cfg.pattern = L.PRECISIONS[precision], L.PATTERNS[pattern]
    elem = {"f64": 8, "f32": 4}.get(precision, 2)
    psi_elem = 8 if precision == "f64" else 4
    sb, pb = L.lbm_required_bytes(cfg)
    state = torch.empty(sb + 16, dtype=torch.uint8, device="cuda")
    psi = torch.empty(pb + 16, dtype=torch.uint8, device="cuda")
    out = []
    for a, b in ((0, 0), (elem, 0), (8, 0), (0, psi_elem), (4 if elem == 2 else elem, 8)):
        cfg.ext_state, cfg.ext_state_bytes = state.data_ptr() + a, sb
        cfg.ext_psi, cfg.ext_psi_bytes = psi.data_ptr() + b, pb
        h = L.lbm_create_ex(cfg)
        try:
            L.lbm_set_option(h, "diag_interval", 2)
            L.lbm_set_populations(h, f0)
            if L.lbm_get_option(h, "fused") and pattern == "ab" and a % 16:
                with pytest.raises(L.LbmError):
                    L.lbm_step(h, 1)
            L.lbm_set_option(h, "fused", 0)
            L.lbm_set_populations(h, f0)
            L.lbm_step(h, 6)
            L.lbm_sync(h)
            m = L.lbm_moments(h, shape[::-1])
            out.append((L.lbm_get_populations(h, shape[::-1]), m, L.lbm_diagnostics(h, True).as_dict()["liquid_count"]))
        finally:
            L.lbm_destroy(h)
    for f, m, n in out[1:]:
        np.testing.assert_array_equal(f, out[0][0])
        for k in m:
            np.testing.assert_array_equal(m[k], out[0][1][k])
        assert n == out[0][2]
    for cfg.ext_state, cfg.ext_psi in ((state.data_ptr() + 1, psi.data_ptr()), (state.data_ptr(), psi.data_ptr() + 2)):
        with pytest.raises(L.LbmError) as ei:
            L.lbm_create_ex(cfg)
        assert "aligned" in str(ei.value)
