"""Rays cut into segments whose elimination that way is given up late or should be: by the system of the segments' last
zones alone, in the launch whose other segments ask whether their ray is still good."""
import numpy as np
import pytest

from oracle import btd as obtd
from vx_inputs import btd as gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-12  # normwise after two refinement sweeps, as for the other systems


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
    x = sv.solve(t["offsets"].to(torch.int32), t["A"], t["B"], t["C"], t["d"]).cpu().numpy()
    ok = sv.check()
    sv.close()
    return x, ok


def _segments(zones, rays):
    """Segments per ray of the first of two levels (the rule of vx_btd_solve)."""
    parts = torch.cuda.get_device_properties(0).multi_processor_count // rays
    while 4 * parts ** 3 > 8.4 * zones ** 2:
        parts -= 1
    return parts


@pytest.mark.parametrize("m", [1, 8, 34, 84])
def test_second_level_alone_fails(m):
    """Tiny blocks in the last zones of a ray's segments: the segments themselves stay small, their system does
    not (its D^-1 C is of order 1e20), and the ray beside it goes on in segments."""
    n = 400
    s = gen.random_system(np.array([n, n]), m, seed=m)
    S = _segments(n, 2)
    tiny = [n + n * (i + 1) // S - 1 for i in range(3, S - 3, 2)]
    for e in tiny:
        s["A"][e], s["C"][e - 1], s["A"][e + 1] = 0.0, 0.0, 0.0
        s["C"][e], s["B"][e] = np.eye(m), 1e-30 * np.eye(m)
    x, ok = _solve(s, m)
    assert ok
    ref = obtd.solve(s["A"], s["B"], s["C"], s["d"], s["offsets"])
    rest = np.setdiff1d(np.arange(n, 2 * n), tiny)
    for z in (np.arange(n), rest, np.array(tiny)):  # (nothing but the tiny zones depends on their x)
        assert np.abs(x[z] - ref[z]).max() <= TOL * np.abs(ref[z]).max()


@pytest.mark.parametrize("n_refine", [0, 1, 2])
@pytest.mark.parametrize("m, seed, kind, scale", [(8, 99, 0, 0.3), (8, 231, 0, 0.1), (20, 10, 1, 1.0), (8, 232, 1, 0.5),
                                                  (4, 28, 1, 1.0), (4, 106, 0, 0.3)])
def test_growth_within_segments(m, seed, kind, scale, n_refine):
    """Random blocks without a dominant diagonal, the entries of D^-1 C and the like between 10 and 90 in the
    segments: alone, the ray is as accurate as among as many rays as the chip takes one block of threads each (the
    same elimination from the first zone on, so the errors agree to a small factor)."""
    n = 150
    g = np.random.default_rng(seed)
    A, B, C = (g.standard_normal((n, m, m)) for _ in range(3))
    A, C = A * scale, C * scale
    B = B + kind * 1.5 * np.sqrt(m) * np.eye(m)
    A[0], C[-1] = 0.0, 0.0
    s = dict(A=A, B=B, C=C, d=g.standard_normal((n, m)), offsets=np.array([0, n], np.int32))
    ref = obtd.solve(A, B, C, s["d"], s["offsets"])
    rays = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    many = {k: np.tile(s[k], (rays,) + (1,) * (s[k].ndim - 1)) for k in ("A", "B", "C", "d")}
    many["offsets"] = np.arange(rays + 1, dtype=np.int32) * n
    err = []
    for q in (s, many):
        x, ok = _solve(q, m, n_refine)
        assert ok
        err.append(np.abs(x[:n] - ref).max() / np.abs(ref).max())
    assert err[0] <= 4 * err[1] + 1e-13, err


def _all_ones():
    return np.array([-1], np.int64).view(np.float64)[0]  # the NaN of memory filled with 0xff


@pytest.mark.parametrize("m, rays, zones", [(1, 3, 3), (8, 3, 5), (33, 3, 4), (20, 2, 60), (84, 1, 150)])
@pytest.mark.parametrize("n_refine", [0, 2])
@pytest.mark.parametrize("block", ["A", "B", "C"])
def test_nan_of_all_ones(m, rays, zones, n_refine, block):
    """One entry of one zone: its ray is NaN and flagged, the others are solved."""
    s = gen.random_system(np.full(rays, zones), m, seed=m)
    z = zones // 2
    s[block][z, m - 1, m // 2] = _all_ones()
    x, ok = _solve(s, m, n_refine)
    assert not ok and np.isnan(x[:zones]).all()
    tol = TOL if n_refine else 1e-4
    for r in range(1, rays):
        a = r * zones
        ref = obtd.solve(s["A"][a:a + zones], s["B"][a:a + zones], s["C"][a:a + zones], s["d"][a:a + zones],
                         np.array([0, zones]))
        assert np.abs(x[a:a + zones] - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("zones", [3, 45])
def test_blocks_below_the_normal_fp32_range(zones):
    """Diagonal blocks between 2^-128 and 2^-126: subnormal FP32 numbers whose reciprocals are finite. They hold
    21 to 23 bits, so a sweep gains about 1e-6, and three leave 1e-12."""
    m = 8
    s = gen.random_system(np.array([zones]), m, seed=zones)
    s["A"][:], s["C"][:] = 0.0, 0.0
    s["B"] *= (2.0 ** -126.1 / np.abs(s["B"]).max(axis=(1, 2)))[:, None, None]
    s["d"] *= 1e-3
    x, ok = _solve(s, m, 3)
    assert ok
    ref = np.linalg.solve(s["B"], s["d"][..., None])[..., 0]
    assert np.abs(x - ref).max() <= TOL * np.abs(ref).max()


@pytest.mark.parametrize("m, lengths", [(5, [1, 2, 0, 7, 1, 9]), (40, [3, 1, 45]), (8, [160]), (84, [44, 1]),
                                        (13, [6] * 200)])
def test_couplings_past_the_ends(m, lengths):
    """A of a ray's first zone and C of its last hold anything at all."""
    s = gen.random_system(lengths, m, seed=m)
    want, ok = _solve(s, m)
    assert ok
    first = s["offsets"][:-1][np.diff(s["offsets"]) > 0]
    last = s["offsets"][1:][np.diff(s["offsets"]) > 0] - 1
    s["A"][first], s["C"][last] = _all_ones(), _all_ones()
    x, ok = _solve(s, m)
    assert ok and np.array_equal(x, want)


@pytest.mark.parametrize("m, zones, min_rays", [(84, 30000, 1), (84, 8000, 31), (84, 8000, 1), (45, 30000, 1), (128, 4000, 1)])
def test_workspace(m, zones, min_rays):
    """Device memory of a handle: per zone what every call needs, and what rays in segments take besides (the header's
    bounds; an array is rounded up to 2 MiB)."""
    from paper_1404_1719_gb300 import BlockTridiagSolver
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    bound = (12 * m * (m + 7) + 4 * (m + 7) + 12 * m + 20) * zones
    if m <= 116 and min_rays <= sms // 5:
        bound += 4 * m * (m + 7) * max(0, 4 * min(zones, 16384) - 3 * zones) + (36 * m * m + 300 * m + 76) * sms
    BlockTridiagSolver(m, 1).close()  # the kernels are loaded
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    sv = BlockTridiagSolver(m, zones, min_rays=min_rays)
    used = before - torch.cuda.mem_get_info()[0]
    sv.close()
    assert used <= bound + 16 * 2 ** 21


@pytest.mark.parametrize("m", [8, 13, 84])
@pytest.mark.parametrize("max_zones, min_rays", [(600, 1), (600, 31), (24000, 1)])
def test_calls_of_any_size(m, max_zones, min_rays):
    """One handle, batches of different zone counts one after the other: whatever an earlier call left in the workspace."""
    from paper_1404_1719_gb300 import BlockTridiagSolver
    sv = BlockTridiagSolver(m, max_zones, min_rays=min_rays)
    for lengths in ([600], [40, 100], [3] * 180, [150], [1], [600], [200, 200, 200]):
        s = gen.random_system(lengths, m, seed=len(lengths) + lengths[0])
        t = {k: torch.from_numpy(np.ascontiguousarray(s[k])).cuda() for k in ("offsets", "A", "B", "C", "d")}
        x = sv.solve(t["offsets"].to(torch.int32), t["A"], t["B"], t["C"], t["d"]).cpu().numpy()
        assert sv.check()
        for a, b in zip(s["offsets"][:-1], s["offsets"][1:]):
            ref = obtd.solve(s["A"][a:b], s["B"][a:b], s["C"][a:b], s["d"][a:b], np.array([0, b - a]))
            assert np.abs(x[a:b] - ref).max() <= TOL * np.abs(ref).max()
    sv.close()


def _fp32_elimination(A, B, C, d, n_refine):
    """Block elimination with an LU factorisation of every block, all in FP32, and refinement from the FP64 residual."""
    from scipy.linalg import lu_factor, lu_solve
    f = np.float32
    a, b, c = A.astype(f), B.astype(f), C.astype(f)
    n, lu, G = len(B), [], []
    for k in range(n):
        lu.append(lu_factor(b[k] - a[k] @ G[-1] if k else b[k]))
        G.append(lu_solve(lu[k], c[k]))
    offsets, x = np.array([0, n]), np.zeros_like(d)
    for _ in range(n_refine + 1):
        r = (d - obtd.apply(A, B, C, x, offsets)).astype(f)
        y = []
        for k in range(n):
            y.append(lu_solve(lu[k], r[k] - a[k] @ y[-1] if k else r[k]))
        for k in range(n - 2, -1, -1):
            y[k] = y[k] - G[k] @ y[k + 1]
        x = x + np.array(y, np.float64)
    return x


@pytest.mark.parametrize("rays", [64, 320])
@pytest.mark.parametrize("m, scale", [(8, 0.3), (8, 1.0), (20, 0.3), (20, 1.0)])
def test_blocks_without_a_dominant_diagonal(m, scale, rays):
    """Random blocks, coupled by 0.3 or all of their size: no further from the solution than block elimination in FP32
    with LU factorisations, in nine rays of ten at least (either error is a random number; with the inverse's own
    error in the solution the median ray was twice as far off, the tenth worst thirty times)."""
    n, sample = 30, 64
    g = np.random.default_rng(m + rays)
    A, B, C = (g.standard_normal((rays * n, m, m)) for _ in range(3))
    A, C = A * scale, C * scale
    A[::n], C[n - 1::n] = 0.0, 0.0
    s = dict(A=A, B=B, C=C, d=g.standard_normal((rays * n, m)), offsets=np.arange(rays + 1, dtype=np.int32) * n)
    for n_refine in (0, 1):
        x, ok = _solve(s, m, n_refine)
        assert ok
        ratio = []
        for r in range(sample):
            z = slice(r * n, r * n + n)
            ref = obtd.solve(A[z], B[z], C[z], s["d"][z], np.array([0, n]))
            e = [np.linalg.norm(q - ref) for q in (x[z], _fp32_elimination(A[z], B[z], C[z], s["d"][z], n_refine))]
            ratio.append(e[0] / e[1])
        assert np.quantile(ratio, 0.9) <= 1.0, (n_refine, np.quantile(ratio, [0.5, 0.9, 1.0]))


@pytest.mark.parametrize("n_refine", [0, 2])
@pytest.mark.parametrize("m, rays, zones", [(2, 60, 7), (8, 2, 150), (8, 100, 12), (33, 60, 9), (84, 1, 60), (128, 3, 6), (20, 320, 5)])
def test_nearly_singular_block(m, rays, zones, n_refine):
    """A zone in a ray's first half whose block's smallest singular value is 1e-6 of the others, in a ray that is well
    conditioned as a whole: no further from the solution than block elimination in FP32 with LU factorisations, in
    the median over the rays (of one ray: within 30 times, what two such eliminations may differ by), and never
    further than solves that gain a factor of 30 each leave, n_refine + 3 of them less one; the other rays are
    solved as ever."""
    s = gen.random_system(np.full(rays, zones), m, seed=m + rays)
    g = np.random.default_rng(m)
    z = [r * zones + zones // 4 for r in range(0, rays, 2)]
    for k in z:
        u, v = (np.linalg.qr(g.standard_normal((m, m)))[0] for _ in range(2))
        size = np.abs(s["B"][k]).max()
        s["B"][k] = size * (u * np.append(np.ones(m - 1), 1e-6)) @ v
        s["A"][k + 1], s["C"][k] = size * np.eye(m), size * np.linalg.qr(g.standard_normal((m, m)))[0]
        s["A"][k] *= 1e-3
        s["C"][k - 1] *= 1e-3
    x, ok = _solve(s, m, n_refine)
    assert ok
    ratio = []
    for r in range(min(rays, 80)):
        a = slice(r * zones, (r + 1) * zones)
        block = [s[q][a] for q in ("A", "B", "C", "d")]
        ref = obtd.solve(*block, np.array([0, zones]))
        err, size = np.abs(x[a] - ref).max(), np.abs(ref).max()
        if r % 2:
            assert err <= (TOL if n_refine else 1e-4) * size, r
        else:
            ratio.append(err / max(np.abs(_fp32_elimination(*block, n_refine) - ref).max(), TOL * size))
            assert err <= max(0.03 ** (n_refine + 2) * size, 30 * err / ratio[-1])
    assert np.median(ratio) <= (1 if len(ratio) > 10 else 30), ratio
