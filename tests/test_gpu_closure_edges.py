"""The electron-gas closure from vanishing to extreme densities and temperatures (both of its
starting ranges and their border), and the chain rule at odd row counts, ragged ends and arrays that are not
16-byte aligned, with the result in place and apart."""
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


@pytest.mark.parametrize("T_log,rho_log", [((-2, 3), (3, 16)), ((-6, 0), (0, 20)), ((3, 9), (-30, 3)), ((-12, -6), (0, 30))])
def test_closure_over_all_magnitudes(T_log, rho_log):
    from paper_1404_1719_gb300 import eos_eta
    rng = np.random.default_rng(5)
    Z = 4097
    s = np.zeros((Z, 4))
    s[:, 0] = 10.0 ** rng.uniform(*T_log, Z)
    s[:, 2] = rng.uniform(0.0, 0.6, Z)
    s[:, 3] = 10.0 ** rng.uniform(*rho_log, Z)
    s[0, 2] = 0.0
    s[1, 3] = 0.0
    st = torch.from_numpy(s).cuda()
    d = eos_eta(st).cpu().numpy()
    e = st[:, 1].cpu().numpy()
    q = 3.0 * np.pi ** 2 * (s[:, 3] * s[:, 2] / 1.66053906660e-24) * (1.973269804e-11 / s[:, 0]) ** 3
    # the cubic is solved to a few roundings of its terms, all of one sign
    lhs = e ** 3 + np.pi ** 2 * e
    assert np.all(np.abs(lhs - q) <= 16 * np.finfo(float).eps * q)
    ok = q > 0
    slope = q[ok] / (3.0 * e[ok] ** 2 + np.pi ** 2)
    for c, v in ((0, -3.0 * slope / s[ok, 0]), (1, slope / s[ok, 2]), (2, slope / s[ok, 3])):
        assert np.all(np.abs(d[ok, c] - v) <= 64 * np.finfo(float).eps * np.abs(v))


@pytest.mark.parametrize("rows", [1, 3, 7, 252])
@pytest.mark.parametrize("Z", [1, 2, 683, 3000])
@pytest.mark.parametrize("shift", [0, 1])
def test_chain_rule_rows_and_alignment(rows, Z, shift):
    from paper_1404_1719_gb300 import eos_chain
    g = torch.Generator("cuda").manual_seed(rows * Z + shift)
    base = torch.randn(Z * rows * 3 + 2, generator=g, dtype=torch.float64, device="cuda")
    jac = base[shift:shift + Z * rows * 3].view(Z, rows, 3)
    deta = torch.randn(Z, 3, generator=g, dtype=torch.float64, device="cuda")
    a, e, y = (jac[..., c].double() for c in range(3))
    D = deta[:, None, :]
    ref = torch.stack([a + e * D[..., 0], y + e * D[..., 1], e * D[..., 2]], -1)
    mag = torch.stack([a.abs() + (e * D[..., 0]).abs(), y.abs() + (e * D[..., 1]).abs(), (e * D[..., 2]).abs()], -1)
    tail = base[shift + Z * rows * 3:].clone()
    res = eos_chain(jac, deta)
    assert torch.all((res - ref).abs() <= 2.0 ** -52 * mag)
    same = eos_chain(jac, deta, out=jac)
    assert torch.equal(same, res) and torch.equal(base[shift + Z * rows * 3:], tail)
