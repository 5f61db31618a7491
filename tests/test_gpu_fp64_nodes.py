"""The FP64 pair kernel's node loop at its edges, against the oracle: odd and even node counts from 2 up, pair
and omega counts that do not divide among the threads, and temperatures on both sides of the border where
2^+-t leaves the FP64 range (q0/2T + |eta| = 690) and the plain loop takes over."""
import numpy as np
import pytest

import oracle
import vx_inputs
from _metrics import magnitudes, worst

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-12  # the FP64 form's tolerance


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_1719_gb300 import _build
    _build.build()
    oracle.build()


@pytest.mark.parametrize("n_bins,n_mu,n_e", [(2, 2, 2), (3, 5, 3), (7, 3, 7), (11, 12, 20), (21, 32, 33), (17, 16, 64), (31, 8, 9)])
def test_fp64_nodes(n_bins, n_mu, n_e):
    from paper_1404_1719_gb300 import PairRates
    e_max = 300.0
    eps = vx_inputs.energy_centres(n_bins, 1.0, e_max)
    st, J, H = vx_inputs.random_zones(24, seed=n_bins + n_e, n_bins=n_bins)
    edge = e_max / 690.0  # T of the border for the largest pair at eta = 0 (q0 / 2 = e_max)
    st[:12, 0] = edge * np.array([0.05, 0.5, 0.98, 0.9999, 1.0001, 1.02, 1.1, 2.0, 8.0, 30.0, 90.0, 1.0])
    st[:12, 1] = [0.0, 5.0, -3.0, 0.0, 0.0, 1.0, 60.0, 79.5, -79.5, -20.0, 0.3, 0.0]
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    rates = PairRates(eps, n_mu, n_e, precision="fp64")
    got = {k: v.cpu().numpy() for k, v in rates.evaluate(dev(st), dev(J), dev(H), phi=True).items()}
    assert rates.check()
    rates.close()
    ref = oracle.evaluate(eps, n_mu, n_e, np.array([0, 1, 2], np.int32), st, J, H, phi=True, mag=True)
    for k in ("j0", "chi0", "j1", "chi1", "phi"):
        g, o, m = got[k], ref[k], magnitudes(ref).get(k)
        if k == "phi":  # production carries e^{-eps_i/T} e^{-eps_j/T}: compared where that factor is a normal number
            cold = 2.0 * e_max / st[:, 0] > 700.0
            g[cold, 0], o[cold, 0] = 0.0, 0.0
        e = worst(g, o, mag=m)
        assert e <= TOL, f"{k}: {e:.3e}"
