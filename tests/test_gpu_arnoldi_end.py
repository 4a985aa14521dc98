"""The end of an Arnoldi iteration in one kernel (norm, Hessenberg column,
rotations, scalars to the host), at its smallest and largest columns and on
both sides of a warp: solves of fixed length against sequential stepping.

Tolerance: the solution of a converged GMRES carries the rounding of L, P^{-1}
and the update, below 1e3 u relative to u, times the amplification of L^{-1}
(at most N = 32 steps of a contraction): 1e-10 leaves three digits."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle as O
from workloads import heat_case_2d

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2002_01108_gb300 import build
    build.build()


@pytest.mark.parametrize("restart,iters", [(1, 40), (2, 40), (32, 32), (33, 33), (60, 60)])
@pytest.mark.parametrize("left", [False, True])
def test_solves_of_fixed_length_reach_the_stepping_solution(restart, iters, left):
    import torch
    from paper_2002_01108_gb300 import Problem
    case = heat_case_2d(seed=9, m=31, N=32, eps=0.05)
    K = O.fd_stiffness(2, case.m, case.a)
    f = O.build_rhs(case.u0, case.fsrc, case.tau)
    ref = O.timestep_solve(f, sp.identity(K.shape[0], format="csr"), K, case.tau)
    with Problem(2, case.m, case.N, T=case.T, max_restart=60) as p:
        p.set_eps(case.eps)
        u, info = p.gmres_solve(torch.from_numpy(f).cuda(), restart=restart, rtol=1e-300, maxit=iters,
                                left_pc=left)
        u = u.cpu().numpy()
    assert info["iters"] <= iters and info["true_relres"] <= 1e-12
    assert float(np.linalg.norm(u - ref) / np.linalg.norm(ref)) <= 1e-10
