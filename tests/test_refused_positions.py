"""A set_positions that fails leaves the handle at no positions: calls that read the geometry return its error, launch
nothing, and work again once a set_positions succeeds."""
import numpy as np
import pytest
import torch

from paper_2603_21835_gb300 import inputs

from . import fake_cudart

ESKIN, EDEVICE = -7, -5


def _calls(G, g, dev="cpu"):
    D, V = torch.zeros(g.nblock, dtype=torch.float64, device=dev), torch.zeros(g.ngrid, dtype=torch.float64, device=dev)
    out = lambda n: torch.zeros(n, dtype=torch.float64, device=dev)
    calls = {}
    for p in (G.FP64, G.FP32, G.F16X3):
        calls[f"rho{p}"] = lambda p=p: g.rho(D, p, out=out(g.ngrid))
        calls[f"vlocal{p}"] = lambda p=p: g.vlocal(V, p, out=out(g.nblock))
        calls[f"force{p}"] = lambda p=p: g.force(D, V, p, out=out(3 * g.natoms))
        calls[f"run{p}"] = lambda p=p: g.run(D, V, p, rho=out(g.ngrid), H=out(g.nblock))
    calls["layout_R"] = g.layout_R
    calls["orbitals"] = lambda: g.orbitals(np.zeros((1, 3)))
    calls["brick_lists"] = g.brick_lists
    calls["set_projectors"] = lambda: g.set_projectors([inputs.si_species()])
    return calls


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return fake_cudart.load(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("cause, code", [("fake_refuse", ESKIN), ("fake_plan_error", EDEVICE)])
def test_no_launch_after_a_refused_geometry(fake, cause, code):
    G, lib = fake
    lib.fake_refuse(0)
    lib.fake_plan_error(0)
    w = inputs.si_workload((1, 1, 1), (16, 16, 16), seed=0)
    g = G.Gint(w.system)
    pos = torch.from_numpy(w.system.pos.copy())
    lib.fake_clear()
    g.rho(torch.zeros(g.nblock, dtype=torch.float64), G.FP64, out=torch.zeros(g.ngrid, dtype=torch.float64))
    assert b"k_fx_eval" in lib.fake_log()  # (so the refusals below are not for want of scratch)
    getattr(lib, cause)(1)
    with pytest.raises(G.GintError) as e:
        g.set_positions(pos + 1.0)
    assert e.value.code == code
    for name, call in _calls(G, g).items():
        lib.fake_clear()
        with pytest.raises(G.GintError) as e:
            call()
        assert e.value.code == code and lib.fake_log() == b"", name
    # going back to the old positions is a rebuild, not the skip of unchanged ones
    getattr(lib, cause)(0)
    lib.fake_clear()
    g.ensure_positions(pos)
    assert b"k_brick_count" in lib.fake_log()
    lib.fake_clear()
    g.rho(torch.zeros(g.nblock, dtype=torch.float64), G.FP64, out=torch.zeros(g.ngrid, dtype=torch.float64))
    assert b"k_fx_eval" in lib.fake_log()
    g.close()


def _rho64(G, lib, g):
    lib.fake_clear()
    g.rho(torch.zeros(g.nblock, dtype=torch.float64), G.FP64, out=torch.zeros(g.ngrid, dtype=torch.float64))
    return lib.fake_log()


def test_scratch_of_the_float64_passes_takes_no_memory_that_others_need(fake):
    """A handle whose buffers fit without the float64 scratch is created without it, and its float64 passes run on the
    CUDA-core kernels; one that loses its buffers in a failed set_positions launches nothing."""
    G, lib = fake
    lib.fake_refuse(0)
    lib.fake_plan_error(0)
    unlimited = 2 ** 63
    w = inputs.si_workload((1, 1, 1), (16, 16, 16), seed=0)
    pos = torch.from_numpy(w.system.pos.copy())
    before = lib.fake_live()
    g = G.Gint(w.system)
    full = lib.fake_live() - before
    assert b"k_fx_eval" in _rho64(G, lib, g)
    g.close()
    assert lib.fake_live() == before
    try:
        lib.fake_limit(before + full - 1)
        g = G.Gint(w.system)
        small = lib.fake_live() - before
        log = _rho64(G, lib, g)
        assert small < full and b"k_fx" not in log and b"k_simt_rho" in log
        # a list that grows to exactly what is left
        n = 4000
        lib.fake_list_entries(n)
        lib.fake_limit(before + small + 8 * (n - 50))
        g.set_positions(pos)
        assert b"k_simt_rho" in _rho64(G, lib, g)
        # ... and beyond it
        lib.fake_list_entries(2 * n)
        with pytest.raises(G.GintError) as e:
            g.set_positions(pos)
        assert e.value.code == -2
        with pytest.raises(G.GintError):
            _rho64(G, lib, g)
        assert lib.fake_log() == b""
        lib.fake_limit(unlimited)
        g.set_positions(pos)
        assert b"k_fx_eval" in _rho64(G, lib, g)
        g.close()
    finally:
        lib.fake_limit(unlimited)
        lib.fake_list_entries(50)
    assert lib.fake_live() == before


def test_no_buffer_for_the_brick_lists_alone(fake):
    """The counting pass's lists (1 KB a brick) lie in the scratch buffer: a handle holds what gint_memory says, and less
    than lists and scratch tiles together."""
    G, lib = fake
    lib.fake_refuse(0)
    lib.fake_plan_error(0)
    w = inputs.si_workload((1, 1, 1), (64, 64, 64), seed=0)
    bricks = 16 * 16 * 8
    before = lib.fake_live()
    lib.fake_tiles(bricks * 200)  # 800 bytes a brick of tiles
    lib.fake_limit(2 ** 63)
    g = G.Gint(w.system)
    try:
        live = lib.fake_live() - before
        assert abs(live - g.memory()) <= 0.01 * live
        # without the float64 scratch: the first limit that admits the handle
        g.close()
        lib.fake_limit(before + live - 1)
        g = G.Gint(w.system)
        small = lib.fake_live() - before
        assert abs(small - g.memory()) <= 0.01 * small
        for _ in range(2):  # kept, not grown, by a rebuild of the same size
            g.set_positions(torch.from_numpy(w.system.pos.copy()))
            assert lib.fake_live() - before == small
        rest = small - bricks * 1024
        g.close()
        lib.fake_tiles(bricks * 1024 // 4)  # tiles of the lists' size
        g = G.Gint(w.system)
        assert lib.fake_live() - before - rest == bricks * 1024
    finally:
        g.close()
        lib.fake_limit(2 ** 63)
        lib.fake_tiles(1000)


def test_handles_without_the_float64_scratch(fake):
    """fp64_scratch=False holds the tiles only; the float64 passes run on the CUDA cores, now and after set_positions."""
    G, lib = fake
    lib.fake_refuse(0)
    lib.fake_plan_error(0)
    w = inputs.si_workload((1, 1, 1), (16, 16, 16), seed=0)
    before = lib.fake_live()
    full = G.Gint(w.system)
    n_full = lib.fake_live() - before
    lean = G.Gint(w.system, fp64_scratch=False)
    n_lean = lib.fake_live() - before - n_full
    assert full.memory() - lean.memory() == n_full - n_lean > 0
    assert b"k_fx_eval" in _rho64(G, lib, full) and b"k_simt_rho" in _rho64(G, lib, lean)
    assert _rho64(G, lib, full).count(b"k_fx_eval") == -(-full.stats()["nbricks"] // full.fp64_batch())
    assert lean.fp64_batch() == 0
    lean.set_positions(torch.from_numpy(w.system.pos.copy()))
    assert b"k_simt_rho" in _rho64(G, lib, lean) and lib.fake_live() - before - n_full == n_lean
    assert lib.gint_create_flags(None, 2, None) == -1
    full.close()
    lean.close()


@pytest.mark.gpu
def test_refused_and_recovered_on_the_gpu():
    from paper_2603_21835_gb300 import gint as G

    w = inputs.si_workload((1, 1, 1), (24, 24, 24), seed=0)
    # a cell with vacuum, so that some pairs have no block
    cell = 3.0 * np.asarray(w.system.cell)
    s = inputs.System(cell=cell, pos=w.system.pos[:2], species=w.system.species[:2], sp=w.system.sp, grid=(24, 24, 24))
    far = s.pos.copy()
    far[1] = far[0] + cell.sum(0) / 2
    s = inputs.System(cell=cell, pos=far, species=s.species, sp=s.sp, grid=s.grid)
    g = G.Gint(s)
    D = torch.randn(g.nblock, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    V = torch.randn(g.ngrid, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    Db = torch.from_numpy(g.dense_to_blocks((lambda M: M + M.T)(g.blocks_to_dense(D.cpu().numpy())))).cuda()
    before = g.rho(Db, G.FP64).clone()
    near = far.copy()
    near[1] = near[0] + 2.0
    with pytest.raises(G.GintError) as e:
        g.set_positions(torch.from_numpy(near).cuda())
    assert e.value.code == ESKIN
    for name, call in _calls(G, g, "cuda").items():
        with pytest.raises(G.GintError) as e:
            call()
        assert e.value.code == ESKIN, name
    g.ensure_positions(torch.from_numpy(far).cuda())
    assert torch.equal(g.rho(Db, G.FP64), before)
    g.vlocal(V, G.F16X3)
    g.sync()
