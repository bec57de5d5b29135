"""The compaction at the edges of its forms: the event list holds 4096 consumed particles (more: the status
scan), a tile looks through 24 of them per particle (more: summed marks), and capacities above 2^20 take
256-thread tiles.  Every particle of one species decays (p = 1 - e^-60 rounds to 1), so the number of
consumed particles is exact; ids, species and counts follow from the oracle's step bit for bit,
positions within 1e-12 L (FP64)."""
import numpy as np
import pytest

import oracle as O
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1107_0270_gb300 as pkg  # noqa: E402
from test_gpu_parity import compare_states, oracle_state_from  # noqa: E402


def decaying(k, others, products, L=2.0, replicas=None):
    """k particles that decay among `others` that do not; species 2 and 3 are products."""
    return W.System(dim=3, L=L, dt=1e-5, seed=5, D=[1.0, 1.0, 0.5, 2.0], n_init=[k, others, 0, 0],
                    pairs=[], decays=[W.Decay(0, 60.0 / 1e-5, products, sigma_place=0.004)], replicas=replicas)


def check_counts(sim, st):
    want = np.zeros((sim.n_replicas, sim.n_species), np.int64)
    np.add.at(want, (st["replica"], st["species"]), 1)
    obs = sim.observables()
    assert np.array_equal(obs["counts"], want)
    assert np.array_equal(sim.count_history(obs["step"], 1)[0], want.sum(axis=0))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("products", [(), (2,), (2, 3)])
@pytest.mark.parametrize("k,others,large", [(1, 0, False), (24, 3000, False), (25, 3000, False), (2048, 1, False),
                                            (4096, 5000, False), (4097, 5000, False), (25, 3000, True),
                                            (4096, 5000, True), (4097, 5000, True)])
def test_exact_numbers_of_consumed_particles(k, others, large, products, precision):
    system = decaying(k, others, products)
    factor = 2.0 if not large else 1.1 * (1 << 20) / (k + others)
    sim = pkg.Simulation(system, precision=precision, capacity_factor=factor)
    assert (sim.info()["capacity"] > (1 << 20)) == large
    for _ in range(2):
        g0 = sim.get_state()
        want, ost = O.step(system, oracle_state_from(g0))
        sim.step()
        g1 = sim.get_state()
        if precision == "fp64":
            compare_states(g1, want, system.L)
        assert np.array_equal(g1["ids"], want.ids) and np.array_equal(g1["species"], want.species)
        assert int(g1["next_id"][0]) == want.next_id
        check_counts(sim, g1)
    sim.close()


@pytest.mark.parametrize("decays", [4094, 4095, 4096])
def test_a_reacting_pair_at_the_end_of_the_event_list(decays):
    # one overlapping absorbing pair reacts with certainty: its two entries end at, straddle or exceed the list
    system = decaying(decays, 100, (2,))
    system.pairs = [W.PairRule(1, 3, 0.01, "abs", 0.0, 2)]
    system.n_init = [decays, 100, 0, 1]
    sim = pkg.Simulation(system, precision="fp64")
    st = sim.get_state()
    x = st["x"].copy()
    b = int(np.flatnonzero(st["species"] == 3)[0])
    a = int(np.flatnonzero(st["species"] == 1)[7])
    x[b] = x[a]
    x[b, 0] = (x[a, 0] + 0.004) % system.L
    sim.set_state(x, st["species"], st["ids"], None, st["next_id"], 0)
    g0 = sim.get_state()
    want, ost = O.step(system, oracle_state_from(g0))
    assert ost["reactions"] == 1 and ost["decays"] == decays
    sim.step()
    g1 = sim.get_state()
    compare_states(g1, want, system.L)
    check_counts(sim, g1)
    sim.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("sizes", [[10, 0, 30, 2000, 3], [1400, 1400, 1400], [1, 4000, 200]])
def test_replicas_of_different_sizes(sizes, precision):
    # tiles that hold several replicas, below and above the event list's length
    system = decaying(0, 0, (2, 3), replicas=[W.Replica(1.0 + 0.1 * r, [k, 7 * r, 0, 0]) for r, k in enumerate(sizes)])
    sim = pkg.Simulation(system, precision=precision)
    g0 = sim.get_state()
    sim.step()
    g1 = sim.get_state()
    for r, rep in enumerate(system.replicas):
        at = g0["replica"] == r
        want, _ = O.step(system, O.State(g0["x"][at].copy(), g0["species"][at].copy(), g0["ids"][at].copy(), 0,
                                         int(g0["next_id"][r]), 0.0), replica=r, L=rep.L)
        got = g1["replica"] == r
        assert np.array_equal(g1["ids"][got], want.ids) and np.array_equal(g1["species"][got], want.species)
        assert int(g1["next_id"][r]) == want.next_id
    check_counts(sim, g1)
    sim.close()


def compaction_us(system):
    sim = pkg.Simulation(system, precision="mixed", step_launch="separate")
    sim.run(4)
    best = min(dict(sim.timed_step())["k_compact"] for _ in range(10))
    sim.close()
    return 1e3 * best


def exchanging(n, kdt, replicas=None):
    # two species that turn into each other: a step consumes the share 1 - e^-kdt of all particles
    return W.System(dim=3, L=2.0, dt=1e-6, seed=3, D=[1.0, 1.0], n_init=[n // 2, n - n // 2], pairs=[],
                    decays=[W.Decay(0, kdt / 1e-6, (1,)), W.Decay(1, kdt / 1e-6, (0,))], replicas=replicas)


def test_a_tile_full_of_events_costs_a_scan_not_a_search():
    # every particle looking through its tile's events: 250 us against 8 without events
    assert compaction_us(exchanging(4000, 30.0)) <= 6.0 * compaction_us(exchanging(4000, 1e-9))


def test_counting_many_events_is_not_one_atomic_each():
    # an atomic on a species' one count per particle: 148 us against 12 without events
    assert compaction_us(exchanging(400_000, 0.5)) <= 5.0 * compaction_us(exchanging(400_000, 1e-9))
