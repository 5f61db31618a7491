"""The FP64 pair kernel where several blocks of threads share a zone: the same bits as one block a zone, with an
invalid zone among them, for numbers of bins and angles whose units divide evenly on the threads (shared) or not, and
the kernel matrices as well; on every repeat, and replayed through a graph."""
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


@pytest.mark.parametrize("n_bins,n_mu,n_e,graph", [(21, 32, 16, False), (21, 32, 16, True), (15, 32, 9, False), (31, 16, 8, False),
                                                   (13, 16, 8, False), (4, 5, 8, False)])
def test_same_bits(n_bins, n_mu, n_e, graph):
    from paper_1404_1719_gb300 import PairRates
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    Z = 8 * sms  # no zone is shared
    st, J, H = vx_inputs.random_zones(Z, seed=n_bins, eta_range=(-5.0, 30.0), n_bins=n_bins)
    st[3, 0] = -1.0  # an invalid zone
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (st, J, H)]
    r = PairRates(vx_inputs.energy_centres(n_bins, 1.0, 300.0), n_mu, n_e, precision="fp64", graph=graph)
    whole = {k: v.clone() for k, v in r.evaluate(*t, phi=True).items()}
    for n in (1, 5, sms // 2, sms, sms + 1, 4 * sms + 1, 5 * sms + 40, 7 * sms + 1):
        part = [x[:n].contiguous() for x in t]
        for _ in range(2):
            for k, v in r.evaluate(*part, phi=True).items():
                assert torch.equal(v.view(torch.int64), whole[k][:n].view(torch.int64)), (n, k)
    r.close()
