"""Few rays, each eliminated from both ends towards the middle, or in segments: rays of one to nine zones and long
ones, a zone whose block cannot be inverted (or only with large numbers in its inverse) where the
elimination from one end can, so that the ray has to be done that way, and a first zone for which nothing
works; against the banded-LU oracle, and around the number of rays from which on one block of threads takes a
ray."""
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


def _in_segments(m):
    """Rays long enough to be cut into segments and, in the same call, ones that are not; with unit couplings
    around a zone whose block is zero or small at the start, inside and at the end of a ray."""
    zones = [1, 2, 3, 7, 8, 9, 40, 99, 100, 101, 100, 100, 100, 100]
    s = gen.random_system(np.array(zones), m, seed=m)
    first = [int(o) for o in s["offsets"]]
    for r, z, f in ((10, 0, 5e-3 / np.abs(s["B"][first[10]]).max()), (11, 30, 0.0), (12, 99, 0.0), (13, 99, 1e-3)):
        k = first[r] + z
        if first[r] < k:
            s["C"][k - 1] = s["A"][k] = np.eye(m)
        if k + 1 < first[r + 1]:
            s["A"][k + 1] = s["C"][k] = np.eye(m)
            s["B"][k + 1] = s["B"][max(k - 1, first[r])]  # nothing cancels in the next zone's block
        s["B"][k] *= f
    s["A"][first[9] + 50:first[9] + 60] = 0.0  # no coupling through a whole segment
    s["C"][first[9] + 49:first[9] + 59] = 0.0
    return s, first


@pytest.mark.parametrize("m", [1, 8, 13, 42, 84, 96, 113, 120])
def test_segments(m):
    s, first = _in_segments(m)
    x, ok = _solve(s, m)
    assert ok
    _close(s, x, range(14))
    s["B"][first[7]] = 0.0  # a ray for which nothing works
    x, ok = _solve(s, m)
    assert not ok
    a, b = first[7], first[8]
    assert np.isnan(x[a:b]).all() and np.isfinite(x[:a]).all() and np.isfinite(x[b:]).all()


@pytest.mark.parametrize("m", [1, 8, 42, 84, 112])
@pytest.mark.parametrize("n_refine", [2, 3])
def test_segments_of_segments(m, n_refine):
    zones = [2, 9, 450, 400]
    s = gen.random_system(np.array(zones), m, seed=m)
    first = [int(o) for o in s["offsets"]]
    s["A"][first[3] + 150:first[3] + 190] = 0.0  # no coupling through whole segments
    s["C"][first[3] + 149:first[3] + 189] = 0.0
    x, ok = _solve(s, m, n_refine)
    assert ok
    _close(s, x, range(4))
    for z in (36, 37, 38, 39, 40, 41, 42, 43, 44, 45, 46, 47):  # whatever the segments: the first zone of one, and others
        s["B"][first[2] + z] = 0.0
        k = first[2] + z
        s["C"][k - 1] = s["A"][k] = s["C"][k] = s["A"][k + 1] = np.eye(m)
    x, ok = _solve(s, m, n_refine)
    assert ok
    _close(s, x, range(4))
