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


# More rows than a grid has blocks along y (65535): rows of several warps, which
# the automatic blocks of two warps would take one at a time.  Even nx in pairs
# and odd in single nodes, both collisions, and the step into padded rows (251
# nodes, from the second step of a replayed graph on).
@pytest.mark.parametrize("shape,precision,pattern,mrt", [
    ((64, 70000, 3), "f64", "ab", 0), ((64, 70000, 3), "f64", "aa", 1), ((128, 70000, 3), "f32", "aa", 0),
    ((256, 65536, 3), "f32", "ab", 0), ((128, 70000, 3), "f16dev", "aa", 1), ((251, 65537, 3), "f32", "ab", 0)])
def test_more_rows_than_a_grid_takes(L, shape, precision, pattern, mrt):
    import torch
    out = []
    for block in (None, (32, 8, 1)):
        with L.Lattice(*shape, 0.9, -5.5, precision=precision, pattern=pattern, block=block, rho_ref=0.1) as lat:
            lat.set_option("collision", mrt)
            if block or shape[0] % 64 == 0:
                lat.set_option("fused", 0)
            lat.init_ligament(5000.0, float(shape[0]), 0.01, 0.3, 2.1, 0.1, 20.0)
            lat.step(4)
            lat.sync()
            n = 19 * shape[0] * shape[1] * shape[2]     # the first array holds the state
            out.append(lat._buffers[0].view({"f64": torch.float64, "f32": torch.float32}.get(precision, torch.float16))[:n].clone())
    assert torch.equal(out[0], out[1])


# A launch that the device refuses (blocks of one node, more rows than a grid
# takes) fails the call, and only that one.
def test_a_refused_launch_fails_one_call(L):
    import torch
    with L.Lattice(4, 70000, 3, 0.9, -5.5, precision="f64", block=(1, 1, 1)) as lat:
        lat.init_ligament(5000.0, 4.0, 0.01, 0.3, 2.1, 0.1, 20.0)
        lat.set_option("graph", 0)
        with pytest.raises(L.LbmError) as ei:
            lat.step(1)
        assert ei.value.status == L.LBM_ERR_CUDA
        torch.zeros(3, device="cuda").add_(1)       # torch checks the last CUDA error
        rho = lat.rho()
        lat.set_option("block_y", 8)
        lat.step(1)
        lat.sync()
        assert abs(lat.rho().sum() / rho.sum() - 1) < 1e-12


# A state brings the densities that tell liquid from vapour: steps recorded
# after loading it use them, replayed or not.
@pytest.mark.parametrize("shape,fused", [((64, 16, 12), 1), ((40, 12, 10), 0)])
@pytest.mark.parametrize("ccl", [0, 1])
def test_loaded_densities_reach_replayed_diagnostics(L, shape, fused, ccl):
    with L.Lattice(*shape, 1.0, -5.3) as lat:
        lat.init_ligament(3.0, float(shape[0]), 0.1, 0.3, 2.1085, 0.0778, 2.0)
        saved = lat.save_state()
    out = []
    for graph in (1, 0):
        with L.Lattice(*shape, 1.0, -5.3) as lat:
            for k, v in (("fused", fused), ("graph", graph), ("diag_ccl", ccl), ("diag_interval", 2)):
                lat.set_option(k, v)
            lat.init_ligament(3.0, float(shape[0]), 0.1, 0.3, 0.3, 0.2, 2.0)
            lat.step(4)
            lat.load_state(saved)
            lat.step(4)
            out.append(lat.diag_history())
    assert out[0] == out[1]
    assert out[0][0]["liquid_volume_w"] != out[0][2]["liquid_volume_w"]


# Where one plane of doubles fits beside the lattice, transfers work (all planes
# together would not fit); what a handle keeps for the next transfer makes room
# for other allocations, of the same handle or another.
def test_transfers_where_one_plane_fits(L, monkeypatch):
    gc.collect()
    shape = (64, 64, 64)                             # a plane takes 2 MiB, 19 planes 38 MiB
    f0 = lbm_inputs.random_populations(*shape, seed=91)
    with L.Lattice(*shape, 0.9, -5.5, precision="f64") as lat:
        monkeypatch.setenv("LBM_ALLOC_CAP_BYTES", str(3 << 20))
        lat.set_populations(f0)
        np.testing.assert_array_equal(lat.populations(), f0)
        one = lat.moments()
        monkeypatch.delenv("LBM_ALLOC_CAP_BYTES")
        all_ = lat.moments()
        np.testing.assert_array_equal(lat.populations(), f0)
    for k in one:
        np.testing.assert_array_equal(one[k], all_[k])


def test_planes_kept_for_transfers_make_room(L, monkeypatch):
    gc.collect()
    shape = (64, 64, 64)
    f0 = lbm_inputs.random_populations(*shape, seed=92)
    with L.Lattice(*shape, 0.9, -5.5) as lat:
        lat.set_populations(f0)
        want = lat.populations()
        monkeypatch.setenv("LBM_ALLOC_CAP_BYTES", str(10 << 20))
        count, _ = lat.droplets()                    # labels: 2 MiB
        lat.set_populations(f0)
        with L.Lattice(32, 32, 32, 0.9, -5.5, torch_buffers=False) as other:   # 5 MiB
            other.set_populations(lbm_inputs.random_populations(32, 32, 32, seed=93))
        np.testing.assert_array_equal(lat.populations(), want)
        assert lat.droplets()[0] == count


# A growth of the diagnostics' scratch or labels that fails leaves the batch
# without them, not with the size they had: smaller instances get their own.
def test_batch_diagnostics_after_a_failed_growth(L, monkeypatch):
    insts = [dict(nx=nx, ny=n, nz=n, tau=0.9, G=-5.5, R0=n / 4.0, lam=float(nx), eps=0.1, phase=0.0, rho_l=2.5,
                  rho_v=0.15, width=2.0) for nx, n in ((8, 8), (64, 32))]
    with L.Batch(insts) as b:
        b.init()
        want = [b.diagnostics(0), b.diagnostics(0, True)]
    with L.Batch(insts) as b:
        b.init()
        assert b.diagnostics(0) == want[0]
        monkeypatch.setenv("LBM_ALLOC_CAP_BYTES", str(1 << 16))    # 2 KB of scratch fit, 157 KB do not
        for ccl in (False, True):
            with pytest.raises(L.LbmError) as ei:
                b.diagnostics(1, ccl)
            assert ei.value.status == L.LBM_ERR_OOM
            assert b.diagnostics(0) == want[0]
        with pytest.raises(L.LbmError):
            b.diagnostics(0, True)                                 # labels for the largest instance
        monkeypatch.delenv("LBM_ALLOC_CAP_BYTES")
        assert b.diagnostics(0, True) == want[1]
        assert b.diagnostics(1, True)["numeric_ok"] == 1


# Asking for in-loop diagnostics with too little memory for the last of their
# buffers fails; asked again with enough, they work.
def test_in_loop_diagnostics_after_a_failed_start(L, monkeypatch):
    gc.collect()
    shape, f0 = (8, 6, 5), lbm_inputs.random_populations(8, 6, 5, seed=94)

    def asked(cap):
        monkeypatch.setenv("LBM_ALLOC_CAP_BYTES", str(cap))
        lat = L.Lattice(*shape, 0.9, -5.5)
        try:
            lat.set_option("diag_interval", 1)
            return lat, True
        except L.LbmError as e:
            assert e.status == L.LBM_ERR_OOM
            return lat, False

    lo, hi = 1 << 10, 1 << 20
    while hi - lo > 1:
        mid = (lo + hi) // 2
        lat, ok = asked(mid)
        lat.close()
        lo, hi = (lo, mid) if ok else (mid, hi)
    lat, ok = asked(lo)
    assert not ok
    monkeypatch.delenv("LBM_ALLOC_CAP_BYTES")
    with lat:
        lat.set_populations(f0)
        lat.set_option("diag_interval", 1)
        lat.step(3)
        assert [r["step"] for r in lat.diag_history()] == [0, 1, 2]


def test_batch_planes_within_the_cap_and_given_back(L, monkeypatch):
    import torch
    gc.collect()
    insts = [dict(nx=64, ny=64, nz=64, tau=0.9, G=-5.5, R0=16.0, lam=64.0, eps=0.1, phase=0.0, rho_l=2.5, rho_v=0.15,
                  width=2.0)]
    monkeypatch.setenv("LBM_ALLOC_CAP_BYTES", str(100 * 64 ** 3))   # pools 80 bytes a node, a plane 8, all planes 152
    with L.Batch(insts, precision="f16dev") as b:
        b.init()
        b.step(2)
        b.diagnostics(0)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        one = b.populations(0)
        assert free - torch.cuda.mem_get_info()[0] < 16 << 20
        monkeypatch.delenv("LBM_ALLOC_CAP_BYTES")
        np.testing.assert_array_equal(b.populations(0), one)
        free = torch.cuda.mem_get_info()[0]
        monkeypatch.setenv("LBM_ALLOC_CAP_BYTES", str(30 << 20))
        with L.Lattice(48, 48, 48, 0.9, -5.5, torch_buffers=False) as lat:      # 17 MiB beside the planes' 38
            lat.set_populations(lbm_inputs.random_populations(48, 48, 48, seed=95))
        assert torch.cuda.mem_get_info()[0] - free > 30 << 20
        np.testing.assert_array_equal(b.populations(0), one)


# A FP64 lattice in exactly the memory it needs: created without the table of
# its pseudo-potential, it computes psi directly.
@pytest.mark.parametrize("rho0", [1.0, 1.3])
def test_f64_lattice_without_room_for_the_psi_table(L, monkeypatch, rho0):
    gc.collect()
    shape, f0 = (12, 9, 8), lbm_inputs.random_populations(12, 9, 8, seed=96)
    cfg = L.lbm_config_default()
    cfg.nx, cfg.ny, cfg.nz, cfg.precision = *shape, L.LBM_F64
    monkeypatch.setenv("LBM_ALLOC_CAP_BYTES", str(sum(L.lbm_required_bytes(cfg)) + 16 + 512))
    out = []
    for cap in (1, 0):
        with L.Lattice(*shape, 0.9, -5.5, precision="f64", rho0=rho0, torch_buffers=False) as lat:
            monkeypatch.delenv("LBM_ALLOC_CAP_BYTES", raising=False)
            lat.set_populations(f0)
            lat.step(5)
            out.append(lat.populations())
    # psi differs by 2e-15 at most (each form's bound); |G| = 5.5 forces of ten
    # psi products each, over 5 steps
    np.testing.assert_allclose(out[0], out[1], rtol=1e-12, atol=1e-14)


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


# Steps whose graph is captured, or whose longer graph is, while the program
# captures a graph of its own on another stream: neither voids the other.
@pytest.mark.parametrize("warm,n", [(0, 20), (20, 400)])
@pytest.mark.parametrize("shape", [(64, 32, 32), (251, 64, 80)])
def test_steps_beside_a_capture_of_the_program(L, shape, warm, n):
    import torch
    main, other = torch.cuda.Stream(), torch.cuda.Stream()
    x = torch.zeros(1000, device="cuda")
    out = []
    for captured in (True, False):
        with torch.cuda.stream(other):
            lat = L.Lattice(*shape, 0.9, -5.5)
        with lat:
            lat.init_ligament(8.0, float(shape[0]), 0.1, 0.3, 2.1, 0.1, 2.0)
            lat.step(warm)
            torch.cuda.synchronize()
            if captured:
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=main):
                    x.add_(1)
                    lat.step(n)
                    x.add_(1)
                g.replay()
            else:
                lat.step(n)
            torch.cuda.synchronize()
            out.append(lat.rho())
    assert float(x.min()) == float(x.max()) == 2.0
    np.testing.assert_array_equal(out[0], out[1])


def test_batch_steps_beside_a_capture_of_the_program(L):
    import torch
    main, other = torch.cuda.Stream(), torch.cuda.Stream()
    insts = [dict(nx=40, ny=20, nz=20, tau=0.9, G=-5.5, R0=5.0, lam=40.0, eps=0.1, phase=0.0, rho_l=2.5, rho_v=0.15,
                  width=2.0)]
    x = torch.zeros(1000, device="cuda")
    out = []
    for captured in (True, False):
        with torch.cuda.stream(other):
            b = L.Batch(insts)
        with b:
            b.init()
            b.step(4)
            torch.cuda.synchronize()
            if captured:
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=main):
                    x.add_(1)
                    b.step(100)          # long enough for the longer graph
                g.replay()
            else:
                b.step(100)
            b.sync()
            out.append(b.populations(0))
    assert float(x.min()) == 1.0
    np.testing.assert_array_equal(out[0], out[1])
