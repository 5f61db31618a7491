"""A zone's rates do not depend on how many zones are in the call: batches on every side of the sizes at
which the kernels change their launch shape give the same bits as one large batch, an invalid zone among
them included."""
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


def _make(kind, n_bins, n_mu, n_e):
    from paper_1404_1719_gb300 import NesRates, PairRates
    eps = vx_inputs.energy_centres(n_bins, 1.0, 300.0)
    if kind == "nes":
        return NesRates(eps, n_mu, n_e)
    if kind == "pair fp64":
        return PairRates(eps, n_mu, n_e, precision="fp64")
    return PairRates(eps, n_mu, n_e, split="split" in kind, precise="precise" in kind)


@pytest.mark.parametrize("kind,n_bins,n_mu,n_e", [("nes", 21, 16, 48), ("nes", 7, 5, 24), ("nes", 17, 12, 15), ("pair", 21, 32, 64),
                                                  ("pair", 5, 3, 20), ("pair split", 17, 16, 48), ("pair precise", 13, 8, 32),
                                                  ("pair fp64", 9, 8, 20)])
def test_same_bits_in_any_batch(kind, n_bins, n_mu, n_e):
    Z = 1400
    st, J, H = vx_inputs.random_zones(Z, seed=n_bins, eta_range=(-5.0, 30.0), n_bins=n_bins)
    st[3, 0] = -1.0  # an invalid zone
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (st, J, H)]
    r = _make(kind, n_bins, n_mu, n_e)
    call = (lambda *x: r.evaluate(*x)) if kind == "pair fp64" else (lambda *x: r.adjoint(*x, forward=True))
    whole = {k: v.clone() for k, v in call(*t).items()}
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for n in (1, 5, sms - 1, 2 * sms, 2 * sms + 1, 7 * sms // 2, 7 * sms // 2 + 1, 760, 1200):
        part = call(*(x[:n].contiguous() for x in t))
        for k, v in part.items():
            assert torch.equal(v.view(torch.int64), whole[k][:n].view(torch.int64)), (kind, n, k)
    with pytest.raises(Exception):
        assert r.check()  # the invalid zone raised the flag
    r.close()
