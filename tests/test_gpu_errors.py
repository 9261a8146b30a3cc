"""Device error bits on their way to the host."""
import numpy as np
import pytest

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
