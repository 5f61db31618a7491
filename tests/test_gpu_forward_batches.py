"""The forward kernel of the mixed form, whose register budget follows the number of zones: a zone's rates have
the same bits in any batch, on either side of one and of two zones per CTA of the larger budget's grid,
and replayed from a captured graph."""
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


@pytest.mark.parametrize("n_bins,n_mu,n_e,opt", [(21, 32, 64, {}), (13, 8, 32, {}), (7, 5, 20, {}), (17, 16, 48, dict(split=True)),
                                                 (9, 8, 32, dict(precise=True)), (13, 8, 32, dict(graph=True))])
def test_same_bits(n_bins, n_mu, n_e, opt):
    from paper_1404_1719_gb300 import PairRates
    Z = 2000
    st, J, H = vx_inputs.random_zones(Z, seed=n_bins, eta_range=(-5.0, 30.0), n_bins=n_bins)
    st[3, 0] = -1.0  # an invalid zone
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (st, J, H)]
    r = PairRates(vx_inputs.energy_centres(n_bins, 1.0, 300.0), n_mu, n_e, **opt)
    whole = {k: v.clone() for k, v in r.evaluate(*t).items()}
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n in (1, sms, 4 * sms, 4 * sms + 1, 6 * sms, 6 * sms + 1, 8 * sms, 8 * sms + 1):
        part = [x[:n].contiguous() for x in t]
        for k, v in r.evaluate(*part).items():
            assert torch.equal(v.view(torch.int64), whole[k][:n].view(torch.int64)), (n, k)
    n = 3 * sms
    part = [x[:n].contiguous() for x in t]
    g = torch.cuda.CUDAGraph()
    if not opt.get("graph"):
        with torch.cuda.graph(g):
            out = r.evaluate(*part)
        for _ in range(2):
            for v in out.values():
                v.zero_()
            g.replay()
            for k, v in out.items():
                assert torch.equal(v.view(torch.int64), whole[k][:n].view(torch.int64)), k
    r.close()
