"""The matching at the edges of its forms: one block takes up to 256 fired pairs and decays together (more:
the grid), a conflict list of 257 to 2048 pairs goes to one block in global memory in 3D (the FP64 2D step
runs every list on the grid).  Pairs that overlap at the start fire with certainty and particles of one
species decay with certainty (p = 1 - e^-60 rounds to 1), so the numbers are exact."""
import math

import numpy as np
import pytest

import oracle as O
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1107_0270_gb300 as pkg  # noqa: E402
from test_gpu_matching import conflict_pairs, greedy_accept  # noqa: E402
from test_gpu_parity import compare_states, oracle_state_from  # noqa: E402

SIGMA = 0.01


def clusters(dim, singles, trios, decays):
    """singles pairs A-B and trios B-A-B that overlap, far from each other, and decaying particles D."""
    n = singles + trios
    m = math.ceil((n + decays) ** (1.0 / dim))
    k = np.arange(n + decays)
    at = np.stack([k % m, (k // m) % m, k // (m * m)] if dim == 3 else [k % m, k // m, 0 * k], axis=1) * 0.2 + 0.1
    if dim == 2:
        at[:, 2] = 0.0
    shift = np.array([0.4 * SIGMA, 0.0, 0.0])
    x = np.concatenate([at[:n], at[:n] + shift, at[singles:n] - shift, at[n:]])
    species = np.repeat(np.array([0, 1, 1, 3], np.int32), [n, n, trios, decays])
    system = W.System(dim=dim, L=0.2 * m, dt=1e-6, seed=9, D=[1.0, 1.0, 0.5, 1.0], n_init=[n, n + trios, 0, decays],
                      pairs=[W.PairRule(0, 1, SIGMA, "abs", 0.0, 2)], decays=[W.Decay(3, 60.0 / 1e-6, (2,))])
    return system, x, species


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("singles,trios,decays", [(256, 0, 0), (257, 0, 0), (0, 128, 0), (1, 128, 0), (100, 40, 76),
                                                  (100, 40, 77), (0, 0, 256), (0, 0, 257), (256, 0, 1)])
def test_exact_numbers_of_pairs_and_decays(singles, trios, decays, precision, dim):
    system, x, species = clusters(dim, singles, trios, decays)
    ids = np.arange(len(x), dtype=np.uint32)
    sim = pkg.Simulation(system, precision=precision)
    sim.set_state(x, species, ids, None, np.array([len(x)], np.uint32), 0)
    g0 = sim.get_state()
    want, ost = O.step(system, oracle_state_from(g0))
    assert ost["fired"] == singles + 2 * trios and ost["decays"] == decays and ost["near_threshold"] == 0
    sim.step()
    g1, f = sim.get_state(), sim.last_fired()
    assert len(f["key"]) == singles + 2 * trios
    acc, _, _ = greedy_accept(f)
    assert np.array_equal(acc, f["accepted"]) and acc.sum() == singles + trios
    if precision == "fp64":
        compare_states(g1, want, system.L)
    # (in the mixed step an FP32 key decides which of a trio's pairs reacts)
    assert np.array_equal(np.sort(g1["species"]), np.sort(want.species)) and int(g1["next_id"][0]) == want.next_id
    sim.close()


@pytest.mark.parametrize("force", [0, 1, 2, 3])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_mid_size_conflict_lists_in_3d(precision, force):
    # 0.4 particles per contact volume at tau = 0.008: about one conflict pair per particle of a species
    n, D = 1000, 0.1
    system = W.System(dim=3, L=(2 * n * 0.005 ** 3 / 0.4) ** (1 / 3), dt=0.008 * 0.005 ** 2 / (2 * D), seed=21,
                      D=[D, D, D], n_init=[n, n, 0], pairs=[W.PairRule(0, 1, 0.005, "abs", 0.0, 2)])
    sim = pkg.Simulation(system, precision=precision, force_paths=force)
    sim.step()
    f = sim.last_fired()
    acc, a, b = greedy_accept(f)
    assert np.array_equal(acc, f["accepted"])
    assert 256 < conflict_pairs(a, b) <= 2048
    sim.close()
