"""A zone's results do not depend on the launch that the number of zones, the grid and the quadrature choose: batches on
either side of each border of the rules give the bits of one large batch."""
import numpy as np
import pytest

import vx_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_1719_gb300 import _build
    _build.build()


def _same_bits(calls, n_bins, Z, sizes, eta=(-5.0, 30.0)):
    st, J, H = vx_inputs.random_zones(Z, seed=n_bins, eta_range=eta, n_bins=n_bins)
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (st, J, H)]
    for call in calls:
        whole = {k: v.clone() for k, v in call(*t).items()}
        for n in sizes:
            for k, v in call(*(x[:n].contiguous() for x in t)).items():
                assert torch.equal(v.view(torch.int64), whole[k][:n].view(torch.int64)), (n, k)


@pytest.mark.parametrize("n_bins,n_mu,n_e", [(25, 16, 48), (25, 12, 36), (21, 16, 48), (17, 12, 36), (13, 16, 48), (21, 8, 24),
                                             (5, 32, 15)])
def test_scattering(n_bins, n_mu, n_e):
    from paper_1404_1719_gb300 import NesRates
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    r = NesRates(vx_inputs.energy_centres(n_bins, 1.0, 300.0), n_mu, n_e)
    borders = (sms, 3 * sms // 2, 2 * sms, 3 * sms, 33 * sms // 10, 7 * sms // 2)
    _same_bits((lambda *x: r.evaluate(*x), lambda *x: r.adjoint(*x, forward=True)), n_bins, 5 * sms,
               [n + d for n in borders for d in (0, 1)])
    assert r.check()
    r.close()


@pytest.mark.parametrize("n_e", [16, 20, 32, 48, 64])
def test_split_tangents(n_e):
    from paper_1404_1719_gb300 import PairRates
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    r = PairRates(vx_inputs.energy_centres(11, 1.0, 300.0), 7, n_e, split=True)
    _same_bits((lambda *x: r.adjoint(*x, forward=True),), 11, 12 * sms, [n + d for n in (4 * sms, 8 * sms) for d in (0, 1)],
               eta=(0.0, 60.0))
    assert r.check()
    r.close()
