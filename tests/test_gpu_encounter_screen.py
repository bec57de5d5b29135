"""The FP64 step compares an encounter draw with an FP32 bound of p_enc first and evaluates p_enc only
below it; the bound must hold for every scaled time tau = D_rel dt / sigma^2.  The scaled distances
carry FP32's rounding of the contact radius, so p_enc's own rounding there grows like 1/sqrt(tau).

Isolated pairs are placed so that their known draw lies 1e-6 below the exact p_enc: every one of them
fires (decisions are exact beyond 1e-9), and a bound that rounding takes below p_enc loses some."""
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

SIGMA, GAP, SPACING = 0.005, 1e-6, 0.04


def _system(dim, tau, n, L, pairs):
    return W.System(dim=dim, L=L, dt=tau * SIGMA ** 2 / 2.0, seed=31, D=[1.0, 1.0, 0.5], n_init=[n, n, 0],
                    pairs=pairs, angle="free_step")


@pytest.mark.parametrize("dim,tau", [(2, 1e-7), (2, 1e-6), (2, 1e-5), (2, 3e-4),
                                     (3, 1e-7), (3, 1e-6), (3, 1e-5), (3, 3e-4), (3, 0.3)])
def test_draws_just_below_p_enc_fire(dim, tau):
    n = 1500
    m = math.ceil(n ** (1.0 / dim))
    L = m * SPACING
    k = np.arange(n)
    centre = np.stack([k % m, (k // m) % m, k // (m * m)], axis=1) * SPACING + 0.5 * SPACING
    if dim == 2:
        centre[:, 1], centre[:, 2] = (k // m) * SPACING + 0.5 * SPACING, 0.0
    species = np.repeat(np.array([0, 1], np.int32), n)
    ids = np.arange(2 * n, dtype=np.uint32)
    rule = [W.PairRule(0, 1, SIGMA, "abs", 0.0, 2)]
    # the free displacements and the encounter draws depend on ids and step only
    free, _ = O.step(_system(dim, tau, n, L, []), O.State(np.concatenate([centre, centre]), species, ids, 0, 2 * n))
    delta = free.x[n:] - free.x[:n]
    delta -= L * np.round(delta / L)
    length = np.linalg.norm(delta, axis=1)
    e = delta / length[:, None]
    near = np.concatenate([centre, centre + SIGMA * 1.0000001 * e])
    _, _, tr = O.step(_system(dim, tau, n, L, rule), O.State(near % L, species, ids, 0, 2 * n), trace=True)
    u = np.zeros(n)
    u[tr["ida"]] = tr["u_enc"]
    assert np.array_equal(np.sort(tr["ida"]), k) and np.array_equal(tr["idb"], tr["ida"] + n)
    # start separations along the displacement, R0 - 1 solved from p_enc(R0 + |delta|, R0) = u + gap
    use = np.flatnonzero((u > 0.01) & (u < 0.9) & (length < 0.25 * SPACING))
    p_enc = (lambda R, R0: O.p_enc3(R, R0, tau)) if dim == 3 else (lambda R, R0: O.p_enc2(R, R0, tau))
    R0 = np.ones(n)
    for q in use:
        lo, hi, step = 0.0, 5.0 * math.sqrt(2.0 * tau), length[q] / SIGMA
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            if p_enc(1.0 + mid + step, 1.0 + mid) > u[q] + GAP:
                lo = mid
            else:
                hi = mid
        R0[q] = 1.0 + lo
    x = np.concatenate([centre, centre + SIGMA * R0[:, None] * e])[np.concatenate([use, use + n])] % L
    sp, pid = species[np.concatenate([use, use + n])], ids[np.concatenate([use, use + n])]
    system = _system(dim, tau, n, L, rule)
    _, ost, tr = O.step(system, O.State(x, sp, pid, 0, 2 * n), trace=True)
    want = set(tr["ida"][tr["fired"] == 1].tolist())
    assert ost["near_threshold"] == 0 and len(use) > 500 and want == set(use.tolist())
    sim = pkg.Simulation(system, precision="fp64")
    sim.set_state(x, sp, pid, None, np.array([2 * n], np.uint32), 0)
    sim.step()
    got = set(sim.last_fired()["id_a"].tolist())
    sim.close()
    assert got == want, f"{len(want - got)} of {len(want)} encounters missed"
