"""The scatter into cell order where a thread takes several particles: systems in which every species
interacts and systems in which some do not, against a grid that gives each particle its own thread."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1107_0270_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("all_interact", [False, True])
def test_several_particles_a_thread(all_interact, precision):
    # 16 blocks of 32 threads an SM: 120 000 particles are more than the grid's threads on any GB300 (at
    # most 160 SMs: 81 920); 256-thread blocks have one each
    system = W.reversible_3d(n_each=100_000, equilibrium_start=True, L=2.0, seed=4)
    system.n_init = [40_000, 40_000, 40_000]
    system.angle = "free_step"
    if all_interact:
        system.pairs = system.pairs + [W.PairRule(2, 2, 0.005, "ref")]
    states = []
    for block in (32, 256):
        sim = pkg.Simulation(system, precision=precision, block_size=block, step_launch="separate")
        sim.run(4)
        states.append((sim.get_state(), sim.observables()["stats"]))
        sim.close()
    (a, sa), (b, sb) = states
    assert sa == sb and sa["fired"] > 100
    for key in ("ids", "species", "x"):
        assert np.array_equal(a[key], b[key]), key


def test_particles_without_a_cell_cost_no_position():
    # 8e6 particles that interact with nothing: only their cell words are read, whatever a position takes
    system = W.System(dim=3, L=2.0, dt=1e-6, seed=3, D=[1.0, 1.0], n_init=[4_000_000, 4_000_000], pairs=[])
    us = {}
    for precision in ("mixed", "fp64"):
        sim = pkg.Simulation(system, precision=precision, step_launch="separate", capacity_factor=1.0)
        sim.run(2)
        us[precision] = 1e3 * min(dict(sim.timed_step())["k_scatter_cells"] for _ in range(10))
        sim.close()
    assert us["fp64"] <= 1.25 * us["mixed"] + 2.0, us
