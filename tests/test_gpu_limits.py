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
