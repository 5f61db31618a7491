"""Host-buffer calls on batches that fit one staging slot and are still cut into chunks: the device calls' bits for
numbers of zones on either side of the second, third and eighth chunk, and partial last chunks."""
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


@pytest.mark.parametrize("autotune", [False, True])
def test_chunks(autotune):
    from paper_1404_1719_gb300 import PairRates
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    five, six = 2 * 5 * sms, 2 * 6 * sms  # zones of a chunk of the tangent and of the forward kernel
    Z = 8 * six + 5
    st, J, H = vx_inputs.random_zones(Z, seed=3, eta_range=(-5.0, 30.0), n_bins=6)
    t = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (st, J, H)]
    r = PairRates(vx_inputs.energy_centres(6, 1.0, 200.0), 4, 16, autotune=autotune)
    whole = {k: v.cpu().numpy() for k, v in r.adjoint(*t, forward=True).items()}
    fwd = {k: v.cpu().numpy() for k, v in r.evaluate(*t).items()}
    for n in (2 * five - 1, 2 * five, 3 * five + 1, 8 * five, Z):
        got = r.adjoint_host(st[:n], J[:n], H[:n], forward=True)
        for k, v in got.items():
            assert np.array_equal(np.asarray(v), whole[k][:n]), (n, k)
    for n in (2 * six - 1, 2 * six, 2 * six + 1, Z):
        got = r.evaluate_host(st[:n], J[:n], H[:n])
        for k, v in got.items():
            assert np.array_equal(np.asarray(v), fwd[k][:n]), (n, k)
    r.close()
