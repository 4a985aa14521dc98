"""The multigrid route's FP64 time transforms in fixed point, at every length
they take and on grids narrower and wider than a tile of 32 (or 16) modes:
P_eps^{-1} against the oracle, with lines of very different size side by side,
and non-finite values.

Tolerance as derived for the FP64 V-cycle: 16 u (log2(N n^2) + 8 levels) / eps
of the largest value."""
import math

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2002_01108_gb300 import build
    build.build()


def case(m, N):
    a = np.exp(np.random.default_rng(75).uniform(-1, 1, (m + 2, m + 2)))
    y = np.random.default_rng(76).uniform(-1, 1, (N, m, m))
    y[:, :, m // 2] *= 1e-9          # a column of small lines between large ones
    y[N // 2:, 0, 0] = 0.0
    return a, y


@pytest.mark.parametrize("m,N,eps", [(7, 32, 0.05), (31, 32, 1e-4), (15, 64, 0.05), (63, 64, 0.05),
                                     (31, 128, 1.0), (15, 256, 0.05), (7, 512, 0.05), (31, 512, 0.05)])
def test_apply_pinv_matches_the_oracle(m, N, eps):
    import torch
    from paper_2002_01108_gb300 import Problem
    a, y = case(m, N)
    with Problem(2, m, N, a_nodes=a, route="mg", precision="fp64", flexible=True) as p:
        p.set_eps(eps)
        z = p.apply_Pinv(torch.from_numpy(y).cuda()).cpu().numpy()
    ref = O.apply_Pinv_mg(y, O.MGHierarchy(O.fd_stiffness_varcoef(a), m), 1.0 / N, eps)
    tol = 16 * U64 * (math.log2(N * (m + 1) ** 2) + 8 * math.log2(m + 1)) / eps
    assert float(np.max(np.abs(z - ref)) / np.max(np.abs(ref))) <= tol


def test_non_finite_values_stay_visible():
    import torch
    from paper_2002_01108_gb300 import Problem
    a, y = case(31, 64)
    with Problem(2, 31, 64, a_nodes=a, route="mg", precision="fp64", flexible=True) as p:
        p.set_eps(0.05)
        for bad in (float("nan"), float("inf")):
            v = y.copy()
            v[3, 4, 5] = bad
            z = p.apply_Pinv(torch.from_numpy(v).cuda()).cpu().numpy()
            assert not np.isfinite(z[:, 4, 5]).any()
