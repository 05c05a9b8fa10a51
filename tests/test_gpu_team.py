"""The three-lane FP64 kernel and the hand-over between the propagate kernels of a call: batches
around the sizes of a team, a warp and one block per SM, batches above the one-lane kernel's lanes
(which pass through every launch), secondaries taken up while they come, budgets that span a
hand-over, and each option of the path, bit for bit against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1410_5323_gb300 import inputs as I
from _parity import assert_bit_identical, by_uid, run_gpu, run_oracle

pytestmark = pytest.mark.gpu
MIX = (("H", .4), ("He", .3), ("N", .2), ("Fe", .1))


def _grid(n, seed):
    return I.kolmogorov_grid(n, 0.25 * I.MPC, 2, 8, 1e-13, seed).astype(np.float32)


def _same(*args, **kw):
    sim, rc = run_gpu(*args, **kw)
    assert rc == 0
    st, orc = run_oracle(*args, **kw)
    assert orc == 0
    assert_bit_identical(sim.state(), st.snapshot())
    return sim


@pytest.mark.parametrize("n", [1, 2, 10, 11, 6081])
def test_batches_around_a_warp_and_a_layer(oracle_lib, n):
    p = I.make_particles(n, n, species=MIX, energy=("power", 1e18, 10 ** 20.5, 2.0))
    _same([_grid(16, 5)], p, I.constant_rate_tables(1 / (200 * I.MPC), 1 / (8 * I.MPC)), 1e-4, I.KPC, I.MPC, 3 * I.MPC,
          seed=n, capacity=56 * n)


@pytest.mark.parametrize("max_steps,calls", [(0, 1), (4, 6)])
def test_batches_above_the_one_lane_kernels_lanes(oracle_lib, max_steps, calls):
    """60 000 nuclei that interact every few steps: one-lane launches, both three-lane launches, and
    budgets whose count goes with a particle that is handed on."""
    n = 60_000
    p = I.make_particles(n, 3, species=MIX, energy=("power", 3e18, 10 ** 20.5, 2.0))
    sim = _same([_grid(16, 6)], p, I.constant_rate_tables(0.0, 1 / (3 * I.MPC)), 1e-4, I.KPC, I.MPC, 2 * I.MPC, seed=9,
                capacity=6 * n, max_steps=max_steps, calls=calls)
    assert sim.counts()["secondaries"] > n // 10


@pytest.mark.parametrize("pickup", [0, 1, 2])
def test_pickup_modes_give_the_same_particles(pickup):
    import paper_1410_5323_gb300 as crp

    p = I.make_particles(2000, 8, species=MIX, energy=("power", 1e18, 10 ** 20.5, 2.0))
    f, t = crp.Field(_grid(16, 7), 0.25 * I.MPC), crp.Tables(I.constant_rate_tables(1 / (300 * I.MPC), 1 / (4 * I.MPC)))
    states = []
    for form in (crp.FORM_FP64, crp.FORM_MIXED):
        for mode in (1, pickup):
            sim = crp.Simulation([f], t, seed=2, capacity=56 * 2000)
            sim.inject(p)
            sim.propagate(1e-4, I.KPC, I.MPC, 8 * I.MPC, form=form, pickup=mode)
            assert sim.sync(60.0) == 0
            states.append(by_uid(sim.state()))
    for a, b in ((0, 1), (2, 3)):
        for k in states[a]:
            assert np.array_equal(states[a][k], states[b][k], equal_nan=states[a][k].dtype.kind == "f"), k


def test_options_small_batch(oracle_lib):
    """Non-power-of-two grids with an origin and negative coordinates, a modulation grid, a reflective
    box, two fields of different realisations."""
    n = 83
    rng = np.random.default_rng(4)
    p = I.make_particles(n, 12, species=(("H", .5), ("Fe", .5)), energy=("power", 1e18, 1e20, 2.0))
    box = ((-2 * I.MPC, -1.5 * I.MPC, 0.0), (4 * I.MPC, 5 * I.MPC, 4.5 * I.MPC))
    p.x[:] = np.asarray(box[0]) + rng.uniform(0.1, 0.9, (n, 3)) * np.asarray(box[1])
    p.grid_id[:] = np.arange(n) % 2
    mods = [np.exp(rng.normal(0.0, 0.4, (6, 5, 7))).astype(np.float32) for _ in range(2)]
    grids = [_grid(18, 13), _grid(18, 14)]
    _same(grids, p, None, 1e-4, I.KPC, I.MPC, 6 * I.MPC, origin=(0.3 * I.MPC, -0.1 * I.MPC, 0.0), mods=mods,
          mod_spacing=0.6 * I.MPC, box=box)


@pytest.mark.parametrize("tables", [False, True])
@pytest.mark.parametrize("n,spare", [(1, 0), (40, 0), (19455, 1), (19457, 0), (300, 40_000)])
def test_precision_form_spread_over_the_device(n, spare, tables):
    """The precision form's launches of one block per SM (small simulations, small lists of large ones,
    and lists just above the limit) against its launches of a fixed shape: the same particles."""
    import paper_1410_5323_gb300 as crp

    p = I.make_particles(n, 21, species=MIX, energy=("power", 1e18, 10 ** 20.5, 2.0))
    f = crp.Field(_grid(16, 8), 0.25 * I.MPC)
    t = crp.Tables(I.constant_rate_tables(1 / (300 * I.MPC), 1 / (20 * I.MPC))) if tables else None
    got = []
    for per_sm in (0, 2):
        sim = crp.Simulation([f], t, seed=4, capacity=(2 * n + 50 if tables else n) + spare)
        sim.inject(p)
        sim.propagate(1e-4, I.KPC, I.MPC, 2 * I.MPC, form=crp.FORM_MIXED, blocks_per_sm=per_sm)
        assert sim.sync(60.0) == 0
        got.append(by_uid(sim.state()))
    for k in got[0]:
        assert np.array_equal(got[0][k], got[1][k], equal_nan=got[0][k].dtype.kind == "f"), k


@pytest.mark.parametrize("n", [400, 9000, 60_000])
def test_no_slot_to_spare(n):
    """As many slots as the run uses: the lists hold secondaries and particles handed on at once."""
    import paper_1410_5323_gb300 as crp

    p = I.make_particles(n, 4, species=MIX, energy=("power", 1e18, 10 ** 20.5, 2.0))
    f, t = crp.Field(_grid(16, 8), 0.25 * I.MPC), crp.Tables(I.constant_rate_tables(0.0, 1 / (2 * I.MPC)))
    states, capacity = [], 30 * n
    for _ in range(2):
        sim = crp.Simulation([f], t, seed=5, capacity=capacity)
        sim.inject(p)
        sim.propagate(1e-4, I.KPC, I.MPC, 3 * I.MPC, form=crp.FORM_FP64)
        assert sim.sync(60.0) == 0
        capacity = n + sim.counts()["secondaries"]
        states.append(by_uid(sim.state()))
    assert capacity > n
    assert_bit_identical(*states)


def test_calls_with_and_without_pickup_on_one_simulation():
    """Lists that a call without pick-ups left full are cleared before the next one looks into them."""
    import paper_1410_5323_gb300 as crp

    p = I.make_particles(3000, 12, species=MIX, energy=("power", 1e18, 10 ** 20.5, 2.0))
    f, t = crp.Field(_grid(16, 9), 0.25 * I.MPC), crp.Tables(I.constant_rate_tables(0.0, 1 / (4 * I.MPC)))
    for form in (crp.FORM_FP64, crp.FORM_MIXED):
        states = []
        for modes in ((1, 1, 1, 1), (1, 0, 2, 0), (0, 1, 0, 2)):
            sim = crp.Simulation([f], t, seed=6, capacity=56 * 3000)
            sim.inject(p)
            for k, mode in enumerate(modes):
                sim.propagate(1e-4, I.KPC, I.MPC, 8 * I.MPC, form=form, pickup=mode, max_steps=4 if k < 3 else 0,
                              order=k % 3)
                if k == 1:
                    sim.reserve(60 * 3000)
            assert sim.sync(60.0) == 0
            states.append(by_uid(sim.state()))
        for s in states[1:]:
            assert_bit_identical(states[0], s)


def test_no_room_for_the_hand_over_and_under_capture(oracle_lib):
    """The first allocation of the first FP64 call fails (the steps of particles handed on): that call
    and a captured one, which must not allocate, finish in the launches that took the particles."""
    import torch

    import paper_1410_5323_gb300 as crp

    n = 60_000
    p = I.make_particles(n, 3, species=MIX, energy=("power", 3e18, 10 ** 20.5, 2.0))
    t = I.constant_rate_tables(0.0, 1 / (3 * I.MPC))
    args = (1e-4, I.KPC, I.MPC, 2 * I.MPC)
    sim = crp.Simulation([crp.Field(_grid(16, 6), 0.25 * I.MPC)], crp.Tables(t), seed=9, capacity=6 * n)
    sim.inject(p)
    try:
        crp.debug_fail_allocations(1)
        sim.propagate(*args, max_steps=4)
    finally:
        crp.debug_fail_allocations(0)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sim.propagate(*args, max_steps=4)
    for _ in range(5):
        graph.replay()
    torch.cuda.synchronize()
    assert sim.sync(60.0) == 0
    st, rc = run_oracle([_grid(16, 6)], p, t, *args, seed=9, capacity=6 * n, max_steps=4, calls=6)
    assert rc == 0
    assert_bit_identical(sim.state(), st.snapshot())


def _run(grid, p, t, args, *, seed, capacity, calls=1, loop=False, **kw):
    import paper_1410_5323_gb300 as crp

    sim = crp.Simulation([crp.Field(grid, 0.25 * I.MPC)], crp.Tables(t), seed=seed, capacity=capacity)
    sim.inject(p)
    for _ in range(calls):
        (sim.propagate_loop if loop else sim.propagate)(*args, **kw)
    assert sim.sync(60.0) == 0
    return sim.state()


@pytest.mark.parametrize("n", [200, 3000, 20_000])
def test_iron_releases_lists_of_every_size(oracle_lib, n):
    """18 nucleons for each iron nucleus: the secondaries' list takes another launch shape than the
    nuclei's, and is above and below what idle lanes take up, in every pick-up mode."""
    import paper_1410_5323_gb300 as crp

    p = I.make_particles(n, 15, species=(("Fe", 1.0),), energy=("power", 10 ** 19.5, 10 ** 20.5, 2.0))
    g, t, args = _grid(16, 10), I.constant_rate_tables(0.0, 1 / (0.1 * I.MPC)), (1e-4, I.KPC, I.MPC, 2 * I.MPC)
    kw = dict(seed=8, capacity=40 * n)
    st, rc = run_oracle([g], p, t, *args, **kw)
    assert rc == 0 and len(st.snapshot()["uid"]) > 12 * n
    plain = _run(g, p, t, args, form=crp.FORM_MIXED, pickup=1, blocks_per_sm=2, **kw)
    for mode in (0, 1, 2):
        assert_bit_identical(_run(g, p, t, args, form=crp.FORM_FP64, pickup=mode, **kw), st.snapshot())
        assert_bit_identical(_run(g, p, t, args, form=crp.FORM_MIXED, pickup=mode, **kw), plain)


@pytest.mark.parametrize("pickup,max_steps,calls", [(0, 0, 1), (0, 4, 6), (2, 0, 1)])
def test_lists_above_twelve_fills_of_the_lanes(oracle_lib, pickup, max_steps, calls):
    """4864 lanes for 60 000 nuclei and their secondaries, which wait for the list's end."""
    p = I.make_particles(60_000, 3, species=MIX, energy=("power", 3e18, 10 ** 20.5, 2.0))
    g, t, args = _grid(16, 6), I.constant_rate_tables(0.0, 1 / (3 * I.MPC)), (1e-4, I.KPC, I.MPC, 2 * I.MPC)
    kw = dict(seed=9, capacity=6 * 60_000, max_steps=max_steps, calls=calls)
    st, rc = run_oracle([g], p, t, *args, **kw)
    assert rc == 0
    assert_bit_identical(_run(g, p, t, args, pickup=pickup, block_size=32, blocks_per_sm=1, **kw), st.snapshot())


@pytest.mark.parametrize("form", [0, 1])
def test_graph_loop_through_every_launch(oracle_lib, form):
    """Slices whose list begins above the lanes and ends below one block per SM, the lists' state kept on
    the device between them: the FP64 form against the oracle, the precision form against calls."""
    n = 90_000
    p = I.make_particles(n, 17, species=MIX, energy=("power", 3e18, 10 ** 20.5, 2.0))
    g, t, args = _grid(16, 6), I.constant_rate_tables(0.0, 1 / (3 * I.MPC)), (1e-4, I.KPC, I.MPC, 2 * I.MPC)
    kw = dict(seed=9, capacity=6 * n)
    got = _run(g, p, t, args, form=form, max_steps=4, loop=True, **kw)
    if form == 0:
        st, rc = run_oracle([g], p, t, *args, **kw)
        assert rc == 0
        assert_bit_identical(got, st.snapshot())
    else:
        assert_bit_identical(got, _run(g, p, t, args, form=form, max_steps=4, calls=60, pickup=1, blocks_per_sm=2, **kw))


def test_queue_full_during_the_hand_over(oracle_lib):
    """Slots run out while particles are handed on: parked ones resume after crp_sim_reserve."""
    import paper_1410_5323_gb300 as crp

    n = 60_000
    p = I.make_particles(n, 18, species=MIX, energy=("power", 3e18, 10 ** 20.5, 2.0))
    g, t, args = _grid(16, 6), I.constant_rate_tables(0.0, 1 / (3 * I.MPC)), (1e-4, I.KPC, I.MPC, 2 * I.MPC)
    sim = crp.Simulation([crp.Field(g, 0.25 * I.MPC)], crp.Tables(t), seed=9, capacity=n + 9000)
    sim.inject(p)
    sim.propagate(*args)
    assert sim.sync(60.0, raise_on_error=False) == crp.api.ERR_QUEUE_FULL
    sim.reserve(6 * n)
    sim.propagate(*args)
    assert sim.sync(60.0) == 0
    st, rc = run_oracle([g], p, t, *args, seed=9, capacity=6 * n)
    assert rc == 0
    assert_bit_identical(sim.state(), st.snapshot())


@pytest.mark.parametrize("tables", [False, True])
@pytest.mark.parametrize("n", [18_240, 18_241, 38_912, 38_913])
def test_batches_around_three_layers_and_the_lanes(oracle_lib, n, tables):
    """One block per SM up to three particles a team, several up to the one-lane kernel's lanes."""
    p = I.make_particles(n, 19, species=MIX, energy=("power", 3e18, 10 ** 20.5, 2.0))
    t = I.constant_rate_tables(1 / (200 * I.MPC), 1 / (3 * I.MPC)) if tables else None
    _same([_grid(16, 5)], p, t, 1e-4, I.KPC, I.MPC, I.MPC, seed=n, capacity=4 * n if tables else n)
