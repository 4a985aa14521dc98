"""The block sums of the Krylov passes: the buffer holds every row that the
largest fused stencil + dots pass writes (up to 32 dots and ||w||^2), and solves
long enough to launch it converge to the stepping solution on the routes whose
rows of L are floating-point (1D, variable coefficient)."""
import os
import shutil
import subprocess

import numpy as np
import pytest
import scipy.sparse as sp

import oracle as O

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_PROGRAM = r"""
#include <cstdio>
#include "bec_internal.h"
int main() {
  using namespace bec;
  long long bad = 0;
  for (long long blocks = 1; blocks < 1LL << 24; blocks = 2 * blocks + 1) {
    for (int nv = 1; nv <= kMaxVec; ++nv)
      // block b < kStencilDotBlocks writes rows 0 .. nv at [row kStencilDotBlocks + b]
      if ((long long)nv * kStencilDotBlocks + kStencilDotBlocks - 1 >= partials_size(blocks)) ++bad;
    if (2 * (blocks - 1) + 1 >= partials_size(blocks)) ++bad;
  }
  std::printf("%lld\n", bad);
  return bad != 0;
}
"""


def test_every_row_of_block_sums_fits(tmp_path):
    cuda = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
    src = tmp_path / "partials.cpp"
    src.write_text(_PROGRAM)
    exe = tmp_path / "partials"
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2002_01108_gb300", "csrc"), "-I", os.path.join(cuda, "include"),
                    str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout.strip() == "0"


@pytest.mark.gpu
@pytest.mark.parametrize("route", ["1d", "mg"])
def test_forty_iterations_in_one_cycle(route):
    """A small diffusion and eps near 1 keep the spectrum spread, so that the
    recurrence goes on past 32 vectors.  Tolerance: the solution of a converged GMRES carries the rounding of L,
    P^{-1} and the update, below 1e3 u relative to u, times the amplification of
    L^{-1} (at most N = 32 steps of a contraction): 1e-10 leaves three digits."""
    import torch
    from paper_2002_01108_gb300 import Problem, build
    build.build()
    m, N = 31, 32
    dim = 1 if route == "1d" else 2
    f = np.random.default_rng(17).uniform(-1, 1, (N,) + (m,) * dim)
    kw = {}
    if route == "mg":
        a = 1e-3 * (1.0 + np.random.default_rng(18).uniform(0, 1, (m + 2, m + 2)))
        kw = dict(route="mg", a_nodes=a)
        K = O.fd_stiffness_varcoef(a)
    else:
        kw = dict(a=1e-3)
        K = O.fd_stiffness(1, m, 1e-3)
    ref = O.timestep_solve(f, sp.identity(K.shape[0], format="csr"), K, 1.0 / N)
    with Problem(dim, m, N, max_restart=60, **kw) as p:
        p.set_eps(0.9)
        u, info = p.gmres_solve(torch.from_numpy(f).cuda(), restart=60, rtol=1e-300, maxit=40)
        u = u.cpu().numpy()
    assert info["iters"] > 32 and info["restarts"] == 0
    assert float(np.linalg.norm(u - ref) / np.linalg.norm(ref)) <= 1e-10
