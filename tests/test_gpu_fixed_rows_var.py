"""The fixed-point rows of L with variable coefficients (2D, multigrid route,
sides from 31): L v and RES against the 5-point rows in extended precision, at
the edges of the warps' tiles (32 columns, 4 rows, the time chunks), for a
varying coefficient and for convection, with values that span many binades,
coefficients that do, and values that are not finite.

Tolerance: the floating-point row's 16 u (1 + 2 k) max|v| with k the largest
diagonal coefficient; where the coefficient jumps by 2^20 from one tile to the
next, the same with each tile's own k."""
import numpy as np
import pytest

import oracle as O
from workloads import circulating_wind_case

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2002_01108_gb300 import build
    build.build()


def rows(v, K, N):
    x = v.reshape(N, -1).astype(np.longdouble)
    C = K.tocoo()
    y = np.zeros_like(x)
    for i in range(N):                          # entry by entry: sparse products are in FP64
        np.add.at(y[i], C.row, C.data.astype(np.longdouble) * x[i, C.col])
    y = x + y / np.longdouble(N)
    y[1:] -= x[:-1]
    return y.reshape(v.shape)


def problem(m, N, kind):
    from paper_2002_01108_gb300 import Problem
    if kind == "wind":
        wind = circulating_wind_case(m, N)[0]
        K = O.fd_convection_diffusion(0.005, wind)[0]
        return Problem(2, m, N, a=0.005, route="mg", wind=wind, side=2.0, mg_smoother="ilu", flexible=True), K
    a = np.exp(np.random.default_rng(5).uniform(-3, 3, (m + 2, m + 2)))
    if kind == "jump":
        a[:, 34:] *= 2.0 ** -20
    return Problem(2, m, N, a_nodes=a, route="mg"), O.fd_stiffness_varcoef(a)


@pytest.mark.parametrize("m,N", [(31, 2), (63, 16), (127, 4), (31, 256)])
@pytest.mark.parametrize("kind", ["flat", "graded", "spike", "wind", "jump"])
def test_L_v_and_RES(m, N, kind):
    import torch
    rng = np.random.default_rng(m + N)
    v = rng.uniform(-1, 1, (N, m, m))
    if kind == "graded":
        v *= 2.0 ** rng.integers(-60, 1, (N, 1, 1)) * 2.0 ** rng.integers(-20, 1, (1, m, m))
    elif kind == "spike":
        v[:] = 0.0
        v[N // 2, m - 1, min(m - 1, 32)] = 3.0
    f = rng.uniform(-1, 1, v.shape)
    p, K = problem(m, N, kind)
    with p:
        y = p.apply_A(torch.from_numpy(v).cuda()).cpu().numpy()
        res = p.true_relres(torch.from_numpy(f).cuda(), torch.from_numpy(v).cuda())
    ref = rows(v, K, N)
    diag = K.diagonal().reshape(m, m) / N
    tol = 16 * U64 * (1 + 2 * diag.max()) * np.max(np.abs(v))
    assert np.max(np.abs(y - ref)) <= tol
    if kind == "jump" and m > 64:              # columns from 64: tiles of small coefficients alone
        low = 16 * U64 * (1 + 2 * diag[:, 64:].max()) * np.max(np.abs(v))
        assert np.max(np.abs(y - ref)[:, :, 64:]) <= low < tol / 16
    want = float(np.linalg.norm((f - ref).ravel().astype(np.float64)) / np.linalg.norm(f))
    assert abs(res - want) <= 1e-12 * want + tol * np.sqrt(v.size) / np.linalg.norm(f)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_values_reach_only_their_neighbours(bad):
    import torch
    m, N = 63, 8
    v = np.random.default_rng(3).uniform(-1, 1, (N, m, m))
    p, K = problem(m, N, "flat")
    clean = rows(v, K, N)
    v[2, 31, 32] = bad                          # the seam of two warps' tiles
    with p:
        y = p.apply_A(torch.from_numpy(v).cuda()).cpu().numpy()
    hit = np.zeros(v.shape, dtype=bool)
    for n, j, i in [(2, 31, 32), (2, 30, 32), (2, 32, 32), (2, 31, 31), (2, 31, 33), (3, 31, 32)]:
        hit[n, j, i] = True
    assert not np.isfinite(y[hit]).any()
    assert np.max(np.abs(y[~hit] - clean[~hit])) <= 16 * U64 * (1 + 2 * K.diagonal().max() / N)
