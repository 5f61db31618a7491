"""The FP64 pair kernel's exponentials by themselves: one pair, two angles and one pair of nodes, in zones so
degenerate that the kernel's entry is a constant times one node's 2^t but for a part in 1e11. 2^t goes by a table
of 2^{j/4096} and a polynomial in the remainder r/4096; where that polynomial's quadratic term would be rounded
to FP32, the entry would be off by a known amount of up to 5e-16, up in some zones and down in others."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_1719_gb300 import _build
    _build.build()


def _zones(Z=200_000, seed=1):
    rng = np.random.default_rng(seed)
    T, eta = rng.uniform(2.3, 4.0, Z), rng.uniform(70.0, 79.0, Z)
    return np.stack([T, eta, np.full(Z, 0.2), np.full(Z, 1e12)], 1)


def _entry(T, eta, eps, cos, tau):
    """The two-node rule of term I at one angle between momenta of energy eps, up to a constant factor."""
    T, eta = T.astype(np.longdouble), eta.astype(np.longdouble)
    y = 1 - cos
    q0, s = 2 * eps, 2 * eps * eps * y
    q = np.sqrt(q0 * q0 - s)
    kq, perp = eps * (q0 - eps * y), eps ** 4 * y * (2 - y) / q ** 2  # k.q (of either momentum), |k_perp|^2
    out = 0
    for t in (tau, -tau):
        E = q0 / 2 + q / 2 * t
        Ec = (2 * q0 * E - s) / (2 * q)
        pk = E * eps - Ec * kq / q
        matrix = pk * s / 2 - (pk * pk - (E * E - Ec * Ec) * perp / 2)
        out = out + matrix / ((1 + np.exp(eta - E / T)) * (1 + np.exp(-eta - (q0 - E) / T)))
    return out


def _fp32_error(T, h, tau):
    """What rounding the quadratic term of 2^{-t}'s polynomial to FP32 adds, relative to 2^{-t}."""
    f = np.float32
    L1 = np.log(2.0) / 4096
    t = (np.longdouble(h) / T.astype(np.longdouble) * tau / np.log(np.longdouble(2)) * 4096)
    r = (t - np.rint(t)).astype(np.float64)
    rf = r.astype(f)
    got = f(f(L1 * L1 / 2) * rf) * rf - f(f(f(L1 ** 3 / 6) * rf) * rf) * rf
    return got.astype(np.float64) - ((L1 * r) ** 2 / 2 - (L1 * r) ** 3 / 6)


def test_quadratic_term_is_not_fp32():
    from paper_1404_1719_gb300 import PairRates
    eps = np.array([100.0, 150.0])
    st = _zones()
    Z = len(st)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    rates = PairRates(eps, 2, 2, precision="fp64")
    J = np.full((Z, 3, 2), 0.25)
    phi = rates.evaluate(dev(st), dev(J), dev(0.5 * J), phi=True)["phi"][:, 1, :, 0, 0].cpu().numpy()
    assert rates.check()
    rates.close()
    tau = 1 / np.sqrt(np.longdouble(3))  # the rule's nodes are +-tau in either variable
    h = np.sqrt(40000 - 20000 * (1 - tau)) / 2
    entry = phi[:, 0] + phi[:, 1] / tau  # twice the part of cos(omega) = tau; the other one, below 2^-8 of it, cancels
    rel = entry / _entry(st[:, 0], st[:, 1], np.longdouble(100), tau, tau)
    rel = (rel / rel.mean() - 1).astype(np.float64)
    assert np.abs(rel).max() < 1e-11
    off = _fp32_error(st[:, 0], h, tau)
    up, down = rel[off > 2.5e-16], rel[off < -2.5e-16]
    assert min(len(up), len(down)) > 2000
    # rounding, the rule's own nodes included, is about 1e-15 a zone, so either mean is known to 2e-17; FP32
    # parts them by 3.6e-16
    assert abs(up.mean() - down.mean()) < 1e-16
