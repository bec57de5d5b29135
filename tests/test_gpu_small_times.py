"""FP64 2D steps at small scaled times tau = D_rel dt / sigma^2: p_enc of every fired pair equals the
oracle's to 1e-11 (the step's bound for it), on both sides of the argument where its I_0 changes form
(Re x = 20, reached below tau of about 1e-2), and a step's cost does not grow as tau falls."""
import time

import pytest

import oracle as O
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1107_0270_gb300 as pkg  # noqa: E402

SIGMA, D = 0.005, 0.1


def crowded(tau, n=1500, bc="abs"):
    return W.System(dim=2, L=(2 * n * SIGMA ** 2 / 0.3) ** 0.5, dt=tau * SIGMA ** 2 / (2 * D), seed=1, D=[D, D, D],
                    n_init=[n, n, 0], pairs=[W.PairRule(0, 1, SIGMA, bc, 0.0, 2)], angle="free_step")


@pytest.mark.parametrize("tau", [1e-6, 1e-5, 1e-4, 1e-3, 3e-3, 1e-2])
def test_fired_pairs_carry_the_exact_p_enc(tau):
    system = crowded(tau, 700)
    sim = pkg.Simulation(system, precision="fp64")
    st = sim.get_state()
    _, ost, tr = O.step(system, O.State(st["x"].copy(), st["species"].copy(), st["ids"].copy(), 0,
                                        int(st["next_id"][0]), 0.0), trace=True)
    sim.step()
    f = sim.last_fired()
    sim.close()
    assert ost["near_threshold"] == 0
    hit = tr["fired"] == 1
    want = {(a, b): p for a, b, p in zip(tr["ida"][hit].tolist(), tr["idb"][hit].tolist(), tr["p_enc"][hit].tolist())}
    got = {(a, b): p for a, b, p in zip(f["id_a"].tolist(), f["id_b"].tolist(), f["p_enc"].tolist())}
    assert len(want) > 50 and want.keys() == got.keys()
    assert max(abs(want[k] - got[k]) for k in want) <= 1e-11


def test_a_step_costs_no_more_at_small_times():
    def seconds(tau):
        sim = pkg.Simulation(crowded(tau, bc="ref"), precision="fp64")
        best = 1e9
        for _ in range(6):
            t = time.perf_counter()
            sim.run(4)
            sim.sync()
            best = min(best, time.perf_counter() - t)
        sim.close()
        return best

    # reflecting pairs, so that the composition stays: a third of the candidates, as many encounters
    assert seconds(1e-5) <= 1.5 * seconds(5e-3)
