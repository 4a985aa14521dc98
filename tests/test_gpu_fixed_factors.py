"""The factor table of the fixed-point time pass, one exponent a tile and frequency,
where the factors span up to 2^23 (eps near 1 and a small diffusion) and where
they are alike: P_eps^{-1} against the oracle."""
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


@pytest.mark.parametrize("dim,m,N", [(2, 31, 32), (2, 63, 256), (2, 31, 1024), (1, 127, 512), (3, 31, 32)])
@pytest.mark.parametrize("eps,a", [(1.0, 1e-5), (1.0, 1.0), (0.9999, 1e-5), (0.05, 1e-2)])
@pytest.mark.parametrize("kind", ["alternating", "flat"])
def test_matches_oracle(dim, m, N, eps, a, kind):
    """Tolerance: the floating-point passes' (test_gpu_fixed_point.py); alternating
    signs put the data at k = N/2, the smallest factor, and leave roundings of the
    sine transforms at frequency 0, which count times the ratio of the factors."""
    import torch
    from paper_2002_01108_gb300 import Problem
    y = np.random.default_rng(m + N).uniform(-1, 1, (N,) + (m,) * dim)
    tau = 1.0 / N
    bound = 16 * U64 * math.log2(N * (m + 1) ** dim) / eps
    if kind == "alternating":
        y = y[:1] * ((-1.0) ** np.arange(N)).reshape((-1,) + (1,) * dim)
        e1, mu = eps ** (1.0 / N), tau * a * dim * math.pi ** 2
        bound *= 1.0 + (1.0 + e1) / (1.0 - e1 + mu)
    with Problem(dim, m, N, a=a, max_restart=2) as p:
        p.set_eps(eps)
        z = p.apply_Pinv(torch.from_numpy(y).cuda())
        torch.cuda.synchronize()
        z = z.cpu().numpy()
    ref = O.apply_Pinv_fst(y, dim, a, tau, eps)
    assert np.max(np.abs(z - ref)) <= bound * np.max(np.abs(ref))
