"""The fixed-point Q1 rows of L (2D, sides from 31): L v and RES against the
9-point stencils in extended precision, at the edges of the warps' tiles (32
columns, 4 rows, the time chunks), where M is small or large beside tau K, with
values that span many binades, and values that are not finite.

Tolerance: the floating-point row's 16 u (sum of |weights|) max|v|."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2002_01108_gb300 import build
    build.build()


def weights(m, N, a):
    h, tau = 1.0 / (m + 1), 1.0 / N
    M = [16.0 * h * h / 36.0, 4.0 * h * h / 36.0, h * h / 36.0]
    K = [8.0 * a / 3.0, -a / 3.0, -a / 3.0]
    return [x + tau * k for x, k in zip(M, K)], M


def rows(v, m, N, a):
    A, M = weights(m, N, a)
    p = np.pad(v.astype(np.longdouble), [(0, 0), (1, 1), (1, 1)])

    def form(w):
        edge = p[:, :-2, 1:-1] + p[:, 2:, 1:-1] + p[:, 1:-1, :-2] + p[:, 1:-1, 2:]
        corner = p[:, :-2, :-2] + p[:, :-2, 2:] + p[:, 2:, :-2] + p[:, 2:, 2:]
        return np.longdouble(w[0]) * p[:, 1:-1, 1:-1] + np.longdouble(w[1]) * edge + np.longdouble(w[2]) * corner
    y, mv = form(A), form(M)
    y[1:] -= mv[:-1]
    return y


def bound(v, m, N, a):
    A, M = weights(m, N, a)
    return 16 * U64 * sum(abs(w[0]) + 4 * abs(w[1]) + 4 * abs(w[2]) for w in (A, M)) * np.max(np.abs(v))


@pytest.mark.parametrize("m,N,a", [(31, 2, 1.0), (31, 64, 1e-7), (63, 16, 1.0), (127, 4, 1e-2), (255, 8, 10.0),
                                   (31, 512, 1e-3)])
@pytest.mark.parametrize("kind", ["flat", "graded", "spike", "zero"])
def test_L_v_and_RES(m, N, a, kind):
    import torch
    from paper_2002_01108_gb300 import Problem
    rng = np.random.default_rng(m + N)
    v = rng.uniform(-1, 1, (N, m, m))
    if kind == "graded":                       # steps and points that span 60 binades
        v *= 2.0 ** rng.integers(-60, 1, (N, 1, 1)) * 2.0 ** rng.integers(-20, 1, (1, m, m))
    elif kind == "spike":
        v[:] = 0.0
        v[N // 2, m - 1, min(m - 1, 32)] = 3.0
    elif kind == "zero":
        v[:] = 0.0
    f = rng.uniform(-1, 1, v.shape)
    with Problem(2, m, N, a=a, space="q1", max_restart=1) as p:
        y = p.apply_A(torch.from_numpy(v).cuda()).cpu().numpy()
        res = p.true_relres(torch.from_numpy(f).cuda(), torch.from_numpy(v).cuda())
    ref = rows(v, m, N, a)
    assert np.max(np.abs(y - ref)) <= bound(v, m, N, a)
    want = float(np.linalg.norm((f - ref).ravel().astype(np.float64)) / np.linalg.norm(f))
    assert abs(res - want) <= 1e-12 * want + bound(v, m, N, a) * np.sqrt(v.size) / np.linalg.norm(f)
    if kind == "zero":
        assert not y.any()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_values_reach_only_their_neighbours(bad):
    import torch
    from paper_2002_01108_gb300 import Problem
    m, N = 63, 8
    v = np.random.default_rng(3).uniform(-1, 1, (N, m, m))
    clean = rows(v, m, N, 1.0)
    v[2, 31, 32] = bad                          # the seam of two warps' tiles
    with Problem(2, m, N, space="q1", max_restart=1) as p:
        y = p.apply_A(torch.from_numpy(v).cuda()).cpu().numpy()
    hit = np.zeros(v.shape, dtype=bool)
    hit[2:4, 30:33, 31:34] = True
    assert not np.isfinite(y[hit]).any()
    assert np.max(np.abs(y[~hit] - clean[~hit])) <= bound(clean * 0 + 1, m, N, 1.0)
