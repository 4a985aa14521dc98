"""The fixed-point finite-difference rows of L (2D and 3D, sides from 31): L v
and RES against the formulas in NumPy, at the edges of the warps' tiles (32
columns, 4 rows, the time chunks), both time schemes, steps whose values differ
by many binades, zeros, and values that are not finite."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2002_01108_gb300 import build
    build.build()


def rows(v, dim, m, N, a, bdf2=False):
    """(L v)^n from the formula of Sec. 2, in extended precision."""
    v = v.astype(np.longdouble)
    c = np.longdouble(a) / N * (m + 1) ** 2
    p = np.pad(v, [(0, 0)] + [(1, 1)] * dim)
    inner = (slice(None),) + (slice(1, -1),) * dim
    lap = 2 * dim * v
    for d in range(1, dim + 1):
        for s in (slice(None, -2), slice(2, None)):
            k = list(inner)
            k[d] = s
            lap = lap - p[tuple(k)]
    prev = np.zeros_like(v)
    prev[1:] = v[:-1]
    if not bdf2:
        return c * lap + v - prev
    prev2 = np.zeros_like(v)
    prev2[2:] = v[:-2]
    return c * lap + 1.5 * v - 2 * prev + 0.5 * prev2


def bound(v, dim, m, N, a):
    """8 u (1 + 2 dim c) max|v|, the bound of the floating-point row (parity tests)."""
    return 8 * U64 * (1 + 2 * dim * a / N * (m + 1) ** 2) * np.max(np.abs(v))


def on_gpu(p, v):
    import torch
    y = p.apply_A(torch.from_numpy(np.ascontiguousarray(v)).cuda())
    torch.cuda.synchronize()
    return y.cpu().numpy()


@pytest.mark.parametrize("dim,m,N,a,scheme", [
    (2, 31, 2, 1.0, "bdf1"), (2, 31, 64, 1e-5, "bdf1"), (2, 63, 16, 1.0, "bdf1"), (2, 127, 4, 0.3, "bdf1"),
    (2, 255, 8, 1.0, "bdf1"), (2, 31, 512, 1.0, "bdf1"), (2, 31, 4, 1.0, "bdf2"), (2, 63, 64, 1e-3, "bdf2"),
    (3, 31, 2, 1.0, "bdf1"), (3, 31, 16, 1e-4, "bdf1")])
@pytest.mark.parametrize("kind", ["flat", "graded", "spike", "zero"])
def test_L_v(dim, m, N, a, scheme, kind):
    from paper_2002_01108_gb300 import Problem
    rng = np.random.default_rng(m + N)
    v = rng.uniform(-1, 1, (N,) + (m,) * dim)
    if kind == "graded":                       # steps and points that span 60 binades
        v *= 2.0 ** rng.integers(-60, 1, (N,) + (1,) * dim) * 2.0 ** rng.integers(-20, 1, (1,) + (m,) * dim)
    elif kind == "spike":
        v[:] = 0.0
        v[N // 2, ..., m - 1] = 3.0            # the last column: an edge lane's neighbour
    elif kind == "zero":
        v[:] = 0.0
    with Problem(dim, m, N, a=a, scheme=scheme, max_restart=1) as p:
        y = on_gpu(p, v)
    ref = rows(v, dim, m, N, a, scheme == "bdf2")
    assert np.max(np.abs(y - ref)) <= bound(v, dim, m, N, a)
    if kind == "zero":
        assert not y.any()


def test_smooth_vector_has_no_bias():
    """On a smooth vector, whose row is small against c v, the mean error over
    the points (which L^{-1} amplifies) stays below a rounding of c max|v|
    divided by the square root of their number (16 of them allowed)."""
    from paper_2002_01108_gb300 import Problem
    m, N = 255, 16
    x = np.sin(np.pi * np.arange(1, m + 1) / (m + 1))
    v = np.exp(-np.arange(N) / N)[:, None, None] * x[:, None] * x
    with Problem(2, m, N, max_restart=1) as p:
        y = on_gpu(p, v)
    e = y - rows(v, 2, m, N, 1.0)
    c = (m + 1) ** 2 / N
    assert abs(float(np.mean(e))) <= 16 * U64 * 4 * c / np.sqrt(v.size)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_values_reach_only_their_neighbours(bad):
    """One value that is not finite changes its own row, its neighbours' rows
    and the next step's; every other row is the finite formula's."""
    from paper_2002_01108_gb300 import Problem
    m, N = 63, 8
    v = np.random.default_rng(3).uniform(-1, 1, (N, m, m))
    clean = rows(v, 2, m, N, 1.0)
    v[2, 31, 32] = bad                          # the seam of two warps' tiles
    with Problem(2, m, N, max_restart=1) as p:
        y = on_gpu(p, v)
    hit = np.zeros(v.shape, dtype=bool)
    for n, j, i in [(2, 31, 32), (2, 30, 32), (2, 32, 32), (2, 31, 31), (2, 31, 33), (3, 31, 32)]:
        hit[n, j, i] = True
    assert not np.isfinite(y[hit]).any()
    assert np.max(np.abs(y[~hit] - clean[~hit])) <= bound(clean * 0 + 1, 2, m, N, 1.0)


def test_relative_residual():
    """RES = ||f - L u|| / ||f|| of a random pair: sums of U squares of rows each
    within the row bound, 16 u log2(U) relative for the sums."""
    import torch
    from paper_2002_01108_gb300 import Problem
    for dim, m, N in ((2, 63, 32), (2, 255, 4), (3, 31, 8)):
        rng = np.random.default_rng(dim)
        f = rng.uniform(-1, 1, (N,) + (m,) * dim)
        u = rng.uniform(-1, 1, f.shape) * 1e-3
        r = f - rows(u, dim, m, N, 1.0)
        ref = float(np.linalg.norm(r.astype(float)) / np.linalg.norm(f))
        with Problem(dim, m, N, max_restart=1) as p:
            res = p.true_relres(torch.from_numpy(f).cuda(), torch.from_numpy(u).cuda())
        assert abs(res - ref) <= 16 * U64 * np.log2(f.size) * ref + bound(u, dim, m, N, 1.0) * np.sqrt(f.size) / np.linalg.norm(f)
