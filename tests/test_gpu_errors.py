"""Device error bits on their way to the host."""
import ctypes as ct

import numpy as np
import pytest

import helpers as H
from oracle import oracle as O
from paper_2402_01181_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import __graft_entry__ as ge
    ge.build()
    from paper_2402_01181_gb300 import mpm
    return mpm


@pytest.mark.parametrize("config", [None, 0, 1, 2, 3, 4])
def test_an_error_of_the_last_substep_reaches_the_readout(M, config):
    """One particle beside the cube runs half a cell a sub-step and leaves the
    grid in the fourth: one CTA sets the bit while the others arrive, and the
    readout of that very call has to report it, time after time."""
    import torch
    sc = scenes.cube8k(2)
    n = sc.n_grid
    x = np.concatenate([sc.x, [[28.75 / n, 20.3 / n, 16.4 / n]]]).astype(np.float32)
    v = np.zeros_like(x)
    v[-1, 0] = 0.5 / n / sc.dt
    xt, vt = torch.tensor(x, device="cuda"), torch.tensor(v, device="cuda")
    out = torch.empty_like(xt)
    sim = M.Sim(M.make_config(n, sc.dt, sc.E, sc.nu, sc.rho, bound=0, max_particles=len(x)))
    if config is not None:
        sim.set_kernel_config(config)
    for k in [3] + [4] * 100:
        sim.load(xt, sc.particle_volume, vt)
        sim.step(k)
        if k == 3:
            sim.read_device(out)
            continue
        with pytest.raises(M.MPMError) as e:
            sim.read_device(out)
        assert e.value.status == M.MPM_ERR_DOMAIN
    sim.close()


@pytest.fixture
def short_wait(monkeypatch):
    """Handles made now give the wait between sub-steps up at its first look."""
    monkeypatch.setenv("GBMPM_WAIT_POLLS", "1")


@pytest.mark.parametrize("config", [None, 2, 3, 4])
def test_a_wait_that_runs_out_stops_what_follows(M, short_wait, config):
    """600 sub-steps are at least two launches: the first one's CTAs lose one
    another, the others do nothing, and the call's successor is refused.  After
    mpm_clear_error only a load helps, and from it single sub-steps (no wait)
    follow the oracle again."""
    sc = H.perturbed_scene(scenes.cube8k(3), seed=4)
    sim = M.sim_from_scene(sc)
    if config is not None:
        sim.set_kernel_config(config)
    assert M.mpm_step(sim.h, 600) == M.MPM_OK
    assert sim.status() == M.MPM_ERR_TIMEOUT
    out = np.empty_like(sc.x)
    assert M.mpm_read_particles(sim.h, out.ctypes.data_as(ct.c_void_p), None, None, None, 0) == M.MPM_ERR_TIMEOUT
    assert M.mpm_step(sim.h, 1) == M.MPM_ERR_TIMEOUT
    sim.clear_error()
    assert M.mpm_step(sim.h, 1) == M.MPM_ERR_STATE
    for _ in range(2):               # the load alone also starts afresh
        sim.load(sc.x, sc.particle_volume, sc.v, sc.F, sc.C)
        for _ in range(3):
            sim.step(1)
        out = sim.read()
        st = O.State(sc.x, sc.v, sc.C, sc.F)
        H.oracle_steps(sc, st, 0, 3)
        assert np.abs(out["x"] - st.x).max() <= 1e-4 * sc.dx and np.abs(out["F"] - st.F).max() <= 1e-5
        assert M.mpm_step(sim.h, 600) == M.MPM_OK and sim.status() == M.MPM_ERR_TIMEOUT
    sim.close()


@pytest.mark.parametrize("checkpoint", [4, 30])
def test_a_rollout_whose_wait_ran_out_is_not_reversed(M, short_wait, checkpoint):
    sc = H.perturbed_scene(scenes.cube8k(3), seed=4, v_scale=0.05, c_scale=0.5, f_dev=0.02)
    sim = M.sim_from_scene(sc)
    for reload in (False, True):
        sim.load(sc.x, sc.particle_volume, sc.v, sc.F, sc.C)
        sim.tape_record(np.zeros((30, 0, 6)), checkpoint)
        if reload:                   # which resets the error bits
            sim.load(sc.x, sc.particle_volume, sc.v, sc.F, sc.C)
        with pytest.raises(M.MPMError) as e:
            sim.tape_backward()
        assert e.value.status == (M.MPM_ERR_STATE if reload else M.MPM_ERR_TIMEOUT)
    sim.close()
