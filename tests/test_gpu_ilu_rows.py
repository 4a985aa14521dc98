"""The row-per-lane ILU smoother of the multigrid route, at the sizes where its
tiling changes: less than a warp of rows, one warp, several warps, both depths
of its operand slots (8 steps ahead, and 4 where 8 do not fit a block), one and
two smoothing steps (the second adds to x).  P_eps^{-1} with one V-cycle a
frequency against the oracle.

Tolerance as derived for the convection-diffusion tests: transforms and level
passes 16 u (log2(N n^2) + 8 levels) / eps, and each of the triangular
recurrences over at most 3 m wavefronts adds 16 u 6 m / eps, once per smoothing
step."""
import math

import numpy as np
import pytest

import oracle as O
from workloads import circulating_wind_case

pytestmark = pytest.mark.gpu

NU = 1.0 / 200.0


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2002_01108_gb300 import build
    build.build()


@pytest.mark.parametrize("precision,m,N,steps", [
    ("fp64", 7, 4, 1), ("fp32", 15, 8, 2), ("fp64", 31, 4, 2), ("fp64", 63, 4, 2), ("fp32", 127, 4, 1),
    ("fp64", 127, 2, 2), ("fp64", 255, 2, 1), ("fp32", 255, 2, 1), ("fp32", 511, 2, 1)])
def test_row_sweeps_match_the_oracle(precision, m, N, steps):
    import torch
    from paper_2002_01108_gb300 import Problem
    eps = 0.05
    wind = circulating_wind_case(m, N)[0]
    K, _ = O.fd_convection_diffusion(NU, wind)
    y = np.random.default_rng(73).uniform(-1, 1, (N, m, m))
    with Problem(2, m, N, a=NU, route="mg", precision=precision, wind=wind, side=2.0,
                 mg_smoother="ilu", flexible=True, mg_pre=steps, mg_post=steps) as p:
        p.set_eps(eps)
        z = p.apply_Pinv(torch.from_numpy(y).cuda()).cpu().numpy()
    ref = O.apply_Pinv_mg(y, O.MGHierarchy(K, m), 1.0 / N, eps, nu1=steps, nu2=steps, smoother="ilu")
    u = 2.0 ** -53 if precision == "fp64" else 2.0 ** -24
    levels = int(math.log2(m + 1))
    tol = 16 * u * (math.log2(N * (m + 1) ** 2) + 8 * levels + 6 * m * steps) / eps
    err = float(np.max(np.abs(z - ref)) / np.max(np.abs(ref)))
    assert err <= tol, (err, tol)
