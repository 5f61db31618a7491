"""The block elimination at its panels' edges (sizes around multiples of 8, 16 and 32) with two CTAs per SM
and shared memory left over from other launches, with couplings that are zero in whole blocks, single
rows and columns, or hold numbers below the FP32 range: against the banded-LU oracle on a few rays, by
the FP64 residual on all, and the same bits on every repeat."""
import numpy as np
import pytest

from oracle import btd as obtd
from vx_inputs import btd as gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-12  # normwise over a ray after two refinement sweeps, as for the other systems
RESID = 1e-13


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_1719_gb300 import _build
    _build.build()


def _system(m, rays, seed):
    rng = np.random.default_rng(seed)
    s = gen.random_system(rng.integers(1, 6, rays), m, seed=seed)
    for q in ("A", "C"):
        M = s[q]
        for z in range(M.shape[0]):
            kind = rng.integers(0, 5)
            if kind == 0:  # one entry per row
                keep = np.zeros((m, m), bool)
                keep[np.arange(m), rng.permutation(m)] = True
                M[z][~keep] = 0.0
            elif kind == 1:  # whole 8 x 8 blocks
                nb = (m + 7) // 8
                M[z][np.kron(rng.random((nb, nb)) < 0.7, np.ones((8, 8), bool))[:m, :m]] = 0.0
            elif kind == 2:  # a single row and a single column
                r, c = rng.integers(0, m, 2)
                v = M[z][r].copy(), M[z][:, c].copy()
                M[z] = 0.0
                M[z][r], M[z][:, c] = v
            elif kind == 3:  # entries that FP32 cannot hold
                M[z][rng.random((m, m)) < 0.5] *= 10.0 ** rng.integers(-320, -40)
    return s


@pytest.mark.parametrize("m", [8, 9, 15, 20, 42, 84, 91, 96])
def test_panels_on_full_chip(m):
    from paper_1404_1719_gb300 import BlockTridiagSolver
    s = _system(m, 320, m)
    t = {k: torch.from_numpy(np.ascontiguousarray(s[k])).cuda() for k in ("offsets", "A", "B", "C", "d")}
    sv = BlockTridiagSolver(m, s["d"].shape[0])
    junk = torch.full((1 << 22,), float("nan"), device="cuda")
    runs = []
    for _ in range(4):
        (junk.sort().values + junk).sum()  # other kernels' shared memory in between
        runs.append(sv.solve(t["offsets"].to(torch.int32), t["A"], t["B"], t["C"], t["d"]))
        assert sv.check()
    sv.close()
    assert all(torch.equal(r, runs[0]) for r in runs)
    x = runs[0].cpu().numpy()
    res = s["d"] - obtd.apply(s["A"], s["B"], s["C"], x, s["offsets"])
    assert np.abs(res).max() <= RESID * max(np.abs(s["d"]).max(), np.abs(s["B"]).max() * np.abs(x).max())
    n = int(s["offsets"][6])
    ref = obtd.solve(s["A"][:n], s["B"][:n], s["C"][:n], s["d"][:n], s["offsets"][:7])
    for r in range(6):
        a, b = s["offsets"][r], s["offsets"][r + 1]
        assert np.abs(x[a:b] - ref[a:b]).max() <= TOL * np.abs(ref[a:b]).max()
