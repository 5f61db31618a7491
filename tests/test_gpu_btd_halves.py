"""Few rays, each eliminated from both ends towards the middle: rays of one to nine zones and long ones, a last
zone whose block cannot be inverted (or only with large numbers in its inverse), so that the elimination
has to go on from the middle outwards, and a first zone for which nothing works; against the banded-LU
oracle, and around the number of rays from which on one block of threads takes a ray."""
import numpy as np
import pytest

from oracle import btd as obtd
from vx_inputs import btd as gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-12  # normwise over a ray after two refinement sweeps, as for the other systems


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_1719_gb300 import _build
    _build.build()


def _solve(s, m, n_refine=2):
    from paper_1404_1719_gb300 import BlockTridiagSolver
    t = {k: torch.from_numpy(np.ascontiguousarray(s[k])).cuda() for k in ("offsets", "A", "B", "C", "d")}
    sv = BlockTridiagSolver(m, s["d"].shape[0], n_refine=n_refine)
    runs = [(sv.solve(t["offsets"].to(torch.int32), t["A"], t["B"], t["C"], t["d"]).cpu().numpy(), sv.check())
            for _ in range(3)]
    sv.close()
    assert all(ok == runs[0][1] and np.array_equal(x, runs[0][0], equal_nan=True) for x, ok in runs)
    return runs[0]


def _close(s, x, rays):
    for r in rays:
        a, b = s["offsets"][r], s["offsets"][r + 1]
        ref = obtd.solve(s["A"][a:b], s["B"][a:b], s["C"][a:b], s["d"][a:b], np.array([0, b - a]))
        assert np.abs(x[a:b] - ref).max() <= TOL * np.abs(ref).max(), r


@pytest.mark.parametrize("m", [1, 13, 84, 96, 128])
def test_last_blocks(m):
    zones = [1, 2, 3, 4, 5, 6, 7, 8, 9, 4, 5, 9, 30, 30, 30]
    s = gen.random_system(np.array(zones), m, seed=m)
    eye = np.eye(m)
    for r in range(9, len(zones)):
        z = int(s["offsets"][r + 1]) - 1
        s["A"][z], s["C"][z - 1] = eye, eye
        s["B"][z] *= (0.0, 1e-3, 1e-30)[r % 3]
    x, ok = _solve(s, m)
    assert ok
    _close(s, x, range(len(zones)))
    bad = 13
    s["B"][s["offsets"][bad]] = 0.0
    x, ok = _solve(s, m)
    assert not ok
    a, b = s["offsets"][bad], s["offsets"][bad + 1]
    assert np.isnan(x[a:b]).all() and np.isfinite(x[:a]).all() and np.isfinite(x[b:]).all()
    _close(s, x, [r for r in range(len(zones)) if r != bad])


@pytest.mark.parametrize("rays, zones", [(75, 9), (152, 9), (153, 9), (190, 40), (191, 40), (304, 40), (305, 40)])
def test_ray_counts(rays, zones):
    m = 20
    rng = np.random.default_rng(rays)
    s = gen.random_system(rng.integers(0, zones, rays), m, seed=rays)
    x, ok = _solve(s, m)
    assert ok
    _close(s, x, [r for r in range(rays) if s["offsets"][r] < s["offsets"][r + 1]])
