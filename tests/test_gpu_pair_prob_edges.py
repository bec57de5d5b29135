"""rd_pair_probs on mixed handles at the ends of FP32: the separations are rounded to FP32 and the
probabilities widened on the integer pipe, so zero, subnormal, huge and exactly-in-contact values are
compared with the FP64 handle's.  Tolerances: p_enc and p_reac 2e-6 absolute (the mixed step's bound);
below FP32's normal range p_enc keeps its magnitude to 1e-4 relative or one subnormal step; every value
is an FP32 number."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1107_0270_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 1027])
def test_extreme_separations(n, offset):
    sigma, tau = 0.005, 0.8
    system = W.reversible_3d(dt=tau * sigma ** 2 / 2.0, n_each=10, L=1.0)
    rng = np.random.default_rng(n)
    # p_enc = exp(-(R-1)^2/tau) over the whole range of FP32 and below, contact, inside, nothing, far
    R = 1.0 + np.sqrt(tau * rng.uniform(0.0, 110.0, n + offset))
    special = [1.0, 0.5, 0.0, 1e-40, 1.0 + np.sqrt(tau * 87.5), 1.0 + np.sqrt(tau * 95.0), 1e6, 1e30]
    R[-min(n, len(special)):] = special[:min(n, len(special))]
    r = torch.tensor(R * sigma, device="cuda")[offset:]
    got = {}
    for precision in ("mixed", "fp64"):
        sim = pkg.Simulation(system, precision=precision)
        pe, pr = sim.pair_probs(r, r)
        got[precision] = pe.cpu().numpy(), pr.cpu().numpy()
        sim.close()
    # the mixed p_reac is a table over the cut-off shell: compared there
    shell = r.cpu().numpy() <= sigma * (1.0 + 5.0 * np.sqrt(2.0 * tau))
    for (g, e), where in zip(zip(got["mixed"], got["fp64"]), (np.ones_like(shell), shell)):
        assert np.array_equal(g, g.astype(np.float32).astype(np.float64))
        assert np.abs(g - e)[where].max(initial=0.0) <= 2e-6
    pe, ref = got["mixed"][0], got["fp64"][0]
    tiny = (ref > 0) & (ref < 1e-37)
    assert np.all(np.abs(pe - ref)[tiny] <= 1e-4 * ref[tiny] + 1.5e-45)
