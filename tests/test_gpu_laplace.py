"""GPU parity of the FP64 pair quantities evaluated from their Laplace transforms, at the ends of their
range: short and long scaled times, starts at and near contact, single pairs and ragged batches.

Tolerances are those of the same quantities elsewhere: propagated vectors 1e-9 (3D) and 1e-8 (2D)
relative (the oracle inverts its own quadratures), p_enc 1e-11 absolute."""
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

SIGMA = 0.005


def pair_system(dim, tau, n=(1, 1, 0), L=1.0, seed=1):
    D = 1.0
    return W.System(dim=dim, L=L, dt=tau * SIGMA ** 2 / (2 * D), seed=seed, D=[D, D, 0.5], n_init=list(n),
                    pairs=[W.PairRule(0, 1, SIGMA, "rad", 0.02 if dim == 3 else 0.01, 2)])


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("tau", [0.02, 0.8, 40.0])
def test_propagate_at_the_ends_of_its_range(dim, tau):
    s = math.sqrt(tau)
    R0 = np.concatenate([[1.0, 1.0 + 1e-9, 1.0 + 1e-3 * s], 1.0 + s * np.linspace(0.05, 3.0, 6)])
    rng = np.random.default_rng([3, dim, int(100 * tau)])
    v = rng.normal(size=(len(R0), 3))
    if dim == 2:
        v[:, 2] = 0.0
    r0 = v / np.linalg.norm(v, axis=1, keepdims=True) * R0[:, None]
    u = rng.uniform(1e-3, 1.0 - 1e-3, size=(len(R0), 4))
    u[0, 0], u[1, 0] = 1e-4, 1.0 - 1e-4
    sim = pkg.Simulation(pair_system(dim, tau), precision="fp64")
    got = sim.propagate(torch.tensor(r0 * SIGMA, device="cuda"), torch.tensor(u, device="cuda")).cpu().numpy() / SIGMA
    sim.close()
    ref = np.array([O.propagate(dim, r0[k], tau, u[k, 0], u[k, 1], u[k, 2]) for k in range(len(u))])
    err = np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() <= (1e-9 if dim == 3 else 1e-8), err


@pytest.mark.parametrize("tau", [0.02, 0.8, 8.0])
def test_fired_pairs_of_a_2d_step_carry_the_exact_p_enc(tau):
    # a crowded 2D box: the step evaluates p_enc only for draws below its closed bound, so the fired
    # set and every fired pair's p_enc must be the oracle's
    n = 150
    L = max(0.12, 12.0 * SIGMA * (1.0 + 5.0 * math.sqrt(2.0 * tau)) / 4.0)
    system = pair_system(2, tau, n=(n, n, 0), L=L, seed=5)
    sim = pkg.Simulation(system, precision="fp64")
    st = sim.get_state()
    state = O.State(st["x"].copy(), st["species"].copy(), st["ids"].copy(), 0, int(st["next_id"][0]), 0.0)
    _, ost, tr = O.step(system, state, trace=True)
    sim.step()
    f = sim.last_fired()
    sim.close()
    assert ost["near_threshold"] == 0
    hit = tr["fired"] == 1
    want = {(a, b): p for a, b, p in zip(tr["ida"][hit].tolist(), tr["idb"][hit].tolist(), tr["p_enc"][hit].tolist())}
    got = {(a, b): p for a, b, p in zip(f["id_a"].tolist(), f["id_b"].tolist(), f["p_enc"].tolist())}
    assert len(want) > 20 and want.keys() == got.keys()
    assert max(abs(want[k] - got[k]) for k in want) <= 1e-11


@pytest.mark.parametrize("precision,n", [("mixed", 1), ("mixed", 129), ("mixed", 300), ("fp64", 1), ("fp64", 33)])
def test_propagated_batch_equals_its_single_pairs(precision, n):
    sim = pkg.Simulation(pair_system(3, 0.8), precision=precision)
    g = torch.Generator(device="cuda").manual_seed(n)
    v = torch.randn(n, 3, dtype=torch.float64, device="cuda", generator=g)
    r0 = v / v.norm(dim=1, keepdim=True) * SIGMA * (1 + torch.rand(n, 1, dtype=torch.float64, device="cuda", generator=g))
    u = torch.rand(n, 4, dtype=torch.float64, device="cuda", generator=g)
    whole = sim.propagate(r0, u)
    for k in {0, n // 2, n - 1}:
        assert torch.equal(sim.propagate(r0[k:k + 1], u[k:k + 1]), whole[k:k + 1])
    sim.close()
