"""Device memory of the mixed handles' p_reac tables: 20 bytes a node (the values and their stencil rows), and
in 3D up to 64 MB of paired rows for the probability batches, which are left out where they would be larger
or the allocator has no room, without a change of any value."""
import math

import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1107_0270_gb300 as pkg  # noqa: E402

SIGMA = 0.005


def system(dim, tau, bc="rad"):
    return W.System(dim=dim, L=2.0, dt=tau * SIGMA ** 2 / 2.0, seed=1, D=[1.0, 1.0, 0.5], n_init=[50, 50, 0],
                    pairs=[W.PairRule(0, 1, SIGMA, bc, 0.02, 2)], angle="free_step")


def nodes(tau):
    # grid of the table: spacing 0.025 min(sqrt(tau), 1) over the cut-off and the propagator's support
    s = math.sqrt(tau)
    h = 0.025 * min(s, 1.0)
    d0 = 5.0 * math.sqrt(2.0) * s + h
    return (math.ceil(d0 / h) + 4) * (math.ceil((d0 + 13.0 * s + 2.0 * h) / h) + 4)


def handle_bytes(system_):
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    sim = pkg.Simulation(system_, precision="mixed")
    used = torch.cuda.memory_allocated() - before
    sim.close()
    return used


@pytest.mark.parametrize("dim,tau", [(2, 0.8), (3, 0.8), (3, 8.0), (3, 9.5), (3, 40.0)])
def test_table_bytes(dim, tau):
    # a reflecting rule has every table of the radiating one but p_reac
    used = handle_bytes(system(dim, tau)) - handle_bytes(system(dim, tau, "ref"))
    paired = 32 * nodes(tau) if dim == 3 and 32 * nodes(tau) <= 64 << 20 else 0
    assert used <= 20 * nodes(tau) + paired + (1 << 20), (used, nodes(tau))


def test_batches_are_the_same_without_paired_rows(monkeypatch):
    tau = 0.8
    g = torch.Generator(device="cuda").manual_seed(3)
    r0 = SIGMA * (1.0 + 6.0 * torch.rand(100_003, dtype=torch.float64, device="cuda", generator=g))
    r = SIGMA * (0.9 + 9.0 * torch.rand(100_003, dtype=torch.float64, device="cuda", generator=g))
    got, refused = [], []
    real = torch.cuda.caching_allocator_alloc
    for room in (True, False):
        def alloc(nbytes, device=None, stream=None):
            if not room and 31 * nodes(tau) < nbytes < 33 * nodes(tau):
                refused.append(nbytes)
                return 0
            return real(nbytes, device, stream)

        monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
        sim = pkg.Simulation(system(3, tau), precision="mixed")
        got.append([t.clone() for t in sim.pair_probs(r0, r)])
        sim.close()
    assert len(refused) == 1
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
