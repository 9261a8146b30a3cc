"""Several sub-steps per launch, the configuration a load chooses, and the
readout and surface kernels at the edges of their warps and words."""
import ctypes as ct

import numpy as np
import pytest

import helpers as H
from oracle import oracle as O
from paper_2402_01181_gb300 import scenes

pytestmark = pytest.mark.gpu

CHOSEN = None            # no configuration set: the load's choice


@pytest.fixture(scope="module")
def M():
    import __graft_entry__ as ge
    ge.build()
    from paper_2402_01181_gb300 import mpm
    return mpm


@pytest.mark.parametrize("config", [CHOSEN, 0, 1, 2, 3, 4])
def test_calls_of_several_lengths_follow_the_oracle(M, config):
    """Calls of 1, 2, 5, 1 and 6 sub-steps (every buffer parity and counter slot
    starts a launch and ends one): the 15 sub-steps within the bounds of 200
    (x to 1e-3 dx, F to 1e-4), the order sorted by block after each call."""
    sc = H.perturbed_scene(scenes.cube8k(3), seed=4)
    sim = M.sim_from_scene(sc)
    if config is not CHOSEN:
        sim.set_kernel_config(config)
    for k in (1, 2, 5, 1, 6):
        sim.step(k)
        ids, keys = sim.read_order()
        x = sim.read()["x"]
        assert np.array_equal(keys, O.block_keys(sc.n_grid, x)[ids]) and np.all(np.diff(keys.astype(np.int64)) >= 0)
        assert np.array_equal(np.sort(ids), np.arange(sc.n))
    out = sim.read()
    sim.close()
    st = O.State(sc.x, sc.v, sc.C, sc.F)
    H.oracle_steps(sc, st, 0, 15)
    assert np.abs(out["x"] - st.x).max() <= 1e-3 * sc.dx
    assert np.abs(out["F"] - st.F).max() <= 1e-4


@pytest.mark.parametrize("n,ppc,grid,threads,ctas_per_sm", [
    (1, 16.0, 32, 512, -32),         # at least 32 CTAs
    (8192, 16.0, 32, 512, -48),      # 8 blocks' worth: a block's chain, the fewest passes, 6 CTAs a block
    (45000, 9.0, 64, 512, 1),        # 78: one CTA per SM at most
    (30000, 3.18, 64, 256, 2),       # 147: a CTA for every block, no spills
    (800000, 9.0, 128, 256, 3),      # 1389, dense
    (50000, 3.2, 64, 128, 4),        # 244, sparse
    (400000, 3.3, 128, 128, 5),      # 1894, sparse
])
def test_load_chooses_by_size_and_density(M, n, ppc, grid, threads, ctas_per_sm):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    x = (0.2 + 0.6 * np.random.default_rng(1).random((n, 3))).astype(np.float32)
    cfg = M.make_config(grid, 1e-5, 1e4, 0.3, 1e3, max_particles=n)
    sim = M.Sim(cfg)
    sim.load(x, 1.0 / (ppc * grid ** 3))
    got = sim.kernel_config()
    assert got == {"config": 0, "threads": threads, "ctas": -ctas_per_sm if ctas_per_sm < 0 else ctas_per_sm * sms}
    sim.set_kernel_config(2)         # a set one is kept by later loads
    sim.load(x, 1.0 / (ppc * grid ** 3))
    assert sim.kernel_config()["config"] == 2 and sim.kernel_config()["threads"] == 128
    sim.close()


@pytest.mark.parametrize("count", [511, 512, 513, 1024, 1025, 4097])
def test_512_threads_single_substep_parity(M, count):
    """Blocks of one, two and more passes of 512 particles, and the run-table
    path of more than four, under a moving capsule."""
    rng = np.random.default_rng(count)
    n = 32
    x = (0.40625 + 0.125 * rng.random((count, 3))).astype(np.float32)
    v, C, F = scenes.random_state(x, count, v_scale=0.3, c_scale=1.0, f_dev=0.05)
    cap = scenes.capsule_shape(0.04, 0.05)
    sc = scenes.Scene("blob", n_grid=n, dt=1e-4, E=2e3, nu=0.3, rho=1e3, x=x, particle_volume=2e-8, v=v, C=C, F=F,
                      friction=0.3,
                      tools=[scenes.Tool(cap, lambda s: np.array([0.47, 0.61 - 1e-4 * (s + 1), 0.46, 0.1, 0.0, 0.2]))])
    sim = M.sim_from_scene(sc)
    assert sim.kernel_config()["threads"] == 512
    ids, _ = sim.read_order()
    start = sim.read()
    sim.set_tool(0, sc.tools[0].pose(0), sc.tools[0].shape)
    sim.step(1)
    out = sim.read()
    ids2, _ = sim.read_order()
    sim.close()
    assert np.array_equal(ids2, O.sorted_order(O.block_keys(n, out["x"]), ids))
    st = H.oracle_state(start)
    mask = H.contact_mask_nodes(sc, st, 0)
    skip = H.particles_touching(mask, st.x, n)
    H.oracle_steps(sc, st, 0, 1, call_len=1)
    assert mask.sum() <= 5
    ok, errs = H.compare_particles(out, st, sc.dx, skip)
    assert ok, errs


@pytest.mark.parametrize("n", [1, 31, 32, 33, 255, 257, 1000])
def test_device_readout_of_any_subset(M, n):
    """A load read back at once is exact, whichever arrays are asked for."""
    import torch
    rng = np.random.default_rng(n)
    x = (0.3 + 0.4 * rng.random((n, 3))).astype(np.float32)
    v, C, F = scenes.random_state(x, n)
    sim = M.Sim(M.make_config(32, 1e-4, 1e4, 0.3, 1e3, max_particles=n + 5))
    sim.load(x, 1e-6, v, F, C)
    for want in ("xvFC", "x", "v", "F", "C", "vF", "xC"):
        t = {k: torch.full((n, c), -7.0, device="cuda") for k, c in (("x", 3), ("v", 3), ("F", 9), ("C", 9))}
        sim.read_device(*[t[k] if k in want else None for k in "xvFC"])
        for k, ref in (("x", x), ("v", v), ("F", F), ("C", C)):
            got = t[k].cpu().numpy()
            assert np.array_equal(got, ref) if k in want else np.all(got == -7.0), (want, k)
    sim.close()


@pytest.mark.parametrize("grid", [8, 16, 32, 64])
@pytest.mark.parametrize("iso", [-1.0, 0.05, 0.5, 1.5, 1e6])
def test_surface_of_scattered_particles(M, grid, iso):
    """Ragged surfaces on rows of less than one, one and two 32-cell words, all
    inside and all outside, against the oracle on the same FP32 density.  With
    exact inputs the two differences and the quotient of an edge point are each
    correctly rounded (3 x 2^-24 of a cell), its sum and product to 2^-23 of the
    unit cube: 4e-7 in all."""
    rng = np.random.default_rng(grid)
    n = 6 * grid * grid
    x = ((0.6 + (grid - 2.2) * rng.random((n, 3))) / grid).astype(np.float32)     # every stencil in the grid
    sc = scenes.Scene("dust", n_grid=grid, dt=1e-5, E=1e3, nu=0.3, rho=1e3, x=x,
                      particle_volume=(1.0 / grid) ** 3 / 3, bound=1)
    sim = M.sim_from_scene(sc)
    field = sim.read_grid()[..., 0] * np.float32(1.0 / (sc.rho * sc.dx ** 3))
    ref = O.surface(field.astype(np.float64), np.float32(iso), sc.dx)
    got = sim.extract_surface(iso)
    dev = sim.extract_surface(iso, device=True).cpu().numpy()
    room = max(1, len(ref) // 2)
    part = np.zeros((room, 3, 3), np.float32)
    count = ct.c_int64()
    M.check(M.mpm_extract_surface(sim.h, 0, iso, part.ctypes.data_as(ct.c_void_p), room, ct.byref(count), 0))
    sim.close()
    assert got.shape == ref.shape and count.value == len(ref)
    assert np.array_equal(got, dev) and np.array_equal(part[:len(ref)], got[:room])
    assert len(ref) == 0 or np.abs(got - ref).max() <= 4e-7
    assert (len(ref) > 0) == (field.min() < iso <= field.max())


def _lattice_sim(M, grid, lo, hi):
    sc = scenes.Scene("lattice", n_grid=grid, dt=2e-5, E=5e3, nu=0.3, rho=1e3,
                      x=scenes.jittered_lattice((lo,) * 3, (hi,) * 3, grid, (2, 2, 2), seed=3),
                      particle_volume=(1.0 / grid) ** 3 / 8)
    return M.sim_from_scene(H.perturbed_scene(sc, seed=4, v_scale=0.05, c_scale=0.5, f_dev=0.02))


def _agree(a, b):
    """The bounds of the segmented backward: 1e-4 of the largest entry."""
    for k in ("E", "nu"):
        assert abs(a[k] - b[k]) <= 1e-4 * abs(a[k]), k
    for k in ("x", "v", "F", "C"):
        ga, gb = a[k].cpu().numpy(), b[k].cpu().numpy()
        assert np.abs(ga - gb).max() <= 1e-4 * np.abs(ga).max(), k


def test_rollout_too_large_to_keep_is_replayed(M):
    """140 sub-steps on a 128^3 grid take 9.4 GB of record, over the 8 GiB that are
    kept: four segments, replayed through two buffers, against one segment,
    which the forward pass records whatever its size."""
    import torch
    out = []
    for ck in (140, 35):
        sim = _lattice_sim(M, 128, 60, 66)
        sim.tape_record(np.zeros((140, 0, 6)), ck)
        g = torch.Generator(device="cuda").manual_seed(5)
        xbar = 1e-4 * torch.randn((sim.n, 3), generator=g, device="cuda")
        out.append(sim.tape_backward(xbar, want_state=True))
        sim.close()
    _agree(*out)


def test_kept_record_serves_a_second_backward_and_the_state_is_the_rollouts_end(M):
    import torch
    sim = _lattice_sim(M, 32, 12, 18)
    sim.tape_record(np.zeros((11, 0, 6)), 4)
    end = sim.read()
    g = torch.Generator(device="cuda").manual_seed(6)
    bars = [1e-3 * torch.randn((sim.n, c), generator=g, device="cuda") for c in (3, 3, 9, 9)]
    first = sim.tape_backward(*bars, want_state=True)
    assert all(np.array_equal(sim.read()[k], end[k]) for k in end)
    sim.step(2)                                  # the record does not depend on the live state
    _agree(first, sim.tape_backward(*bars, want_state=True))
    assert all(np.array_equal(sim.read()[k], end[k]) for k in end)
    one = _lattice_sim(M, 32, 12, 18)
    one.tape_record(np.zeros((11, 0, 6)), 11)
    _agree(one.tape_backward(*bars, want_state=True), first)
    one.close()
    sim.close()
